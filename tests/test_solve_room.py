"""Device memory of handles on the assembled trace matrix (no GPU call): a system whose solves are one
launch holds what crosses blocks in the bytes of its Krylov basis -- at least 8 FP32 or 6 FP64 vectors,
however short the restart -- and a larger system its restart + 1 basis vectors alone."""
import pytest

hd = pytest.importorskip("paper_1711_02751_gb300.hdgdg")


def _bytes(N, k, m, **kw):
    return hd.bytes_required(hd.make_config(N, k, 1e-3, krylov_restart=m, **kw))


@pytest.mark.parametrize("kw,size,room", [(dict(precision="mixed"), 4, 8), ({}, 8, 6)])
@pytest.mark.parametrize("boundary", ["periodic", "wall"])
def test_only_one_launch_solves_hold_exchange_room(kw, size, room, boundary):
    k = 3
    for N, one_launch in ((32, True), (512, False)):
        edges = 2 * N * (N + (boundary == "wall"))
        vector = edges * 3 * (k + 1) * size
        grown = _bytes(N, k, room - 1, boundary=boundary, **kw) - _bytes(N, k, 1, boundary=boundary, **kw)
        per = grown / vector
        if one_launch:
            assert per < room - 2                          # (the reductions' scratch alone)
        else:
            assert room - 2 <= per < room - 1
