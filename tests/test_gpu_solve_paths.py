"""The two paths of the assembled trace solve -- one cooperative launch, and a launch per operation, which
larger systems take -- chosen by hdgdg_set_solve_blocks, so that small systems reach both.

On the launch-per-operation path: the pipelined FP32 product (spmv_kernel = 1: bulk copies into shared
memory, two stages on mbarriers, persistent blocks) against the default one, whole steps bit for bit, at
sizes that give every block several tiles, with a ragged last one (k = 2: 28 edges a tile) and with walls;
and whole-step graphs against host-driven steps, bit for bit, over enough steps for the history to fill.
Between the paths, and between grids: the same trajectory to the solver's tolerance (1e-9 of g a stage
solve in the mixed form, whose states are held to 1e-6; 1e-12 in the FP64 form, held to 1e-9)."""
import numpy as np
import pytest

from oracle import swe
from paper_1711_02751_gb300 import workloads as W

from _common import dt_of, user_state

pytestmark = pytest.mark.gpu
hd = pytest.importorskip("paper_1711_02751_gb300.hdgdg")

ASSEMBLED = dict(precision="mixed", local_precision="f32x2", residual_f32x2=True)


def _large(N, k, boundary="periodic"):
    x, y = hd.node_coords(N, k, boundary=boundary)
    h, hu, hv, b = W.large_state(x, y, seed=11)
    if boundary != "periodic":
        hu, hv = 0.0 * hu, 0.0 * hv
    return h, hu, hv, b, W.advective_dt(x, h, hu, hv, N)


def _run(N, k, init, steps, blocks, **kw):
    h, hu, hv, b, dt = init
    with hd.Sim(N, k, dt, bottom=b, **kw) as s:
        s.set_solve_blocks(blocks)
        s.set_state(h, hu, hv)
        orders = []
        for _ in range(steps):
            s.step(1)
            orders.append(s.stats()["last_guess_order"])
        return s.get_state(), s.stats(), orders


@pytest.mark.parametrize("N,k,boundary", [(96, 3, "periodic"), (128, 2, "periodic"), (40, 1, "wall"),
                                          (24, 4, "periodic"), (160, 2, "periodic"), (47, 4, "wall")])
def test_streamed_product_bit_identical(N, k, boundary):
    init = _large(N, k, boundary)
    runs = [_run(N, k, init, 3, 0, precision="mixed", boundary=boundary, spmv_kernel=kernel) for kernel in (0, 1)]
    one = _run(N, k, init, 3, -1, precision="mixed", boundary=boundary)
    for a, c in zip(runs[0][0], runs[1][0]):
        assert np.array_equal(a, c)
    assert runs[0][1]["krylov_iterations"] == runs[1][1]["krylov_iterations"]
    if N < 160:   # both arms really launched each operation
        assert min(r[1]["kernel_launches"] for r in runs) > one[1]["kernel_launches"] + runs[0][1]["krylov_iterations"]


@pytest.mark.parametrize("name,N,k,kind,steps,kw", [
    ("fp64", 16, 3, "large", 9, {}),
    ("mixed_assembled", 16, 3, "large", 9, ASSEMBLED),
    ("mixed_fp64_local", 12, 2, "large", 7, dict(precision="mixed")),
    ("ars3", 10, 3, "large", 7, dict(scheme="ars3")),
    ("linear_only", 8, 3, "standing", 6, dict(linear_only=True)),
    ("bump8_stiff_guess3", 8, 2, "bump8", 8, dict(krylov_guess=3)),
    ("mixed_assembled_ls_guess2", 12, 3, "large", 7, dict(ASSEMBLED, krylov_guess_ls=True, krylov_guess=2)),
    ("mixed_once", 16, 2, "large", 7, dict(ASSEMBLED, krylov_ortho=1, krylov_restart=5)),
])
def test_graph_steps_equal_host_driven_steps_launch_per_operation(name, N, k, kind, steps, kw):
    m, h, hu, hv, b = user_state(N, k, kind)
    init = (h, hu, hv, b, dt_of(m, h, hu, hv))
    a, sa, ga = _run(N, k, init, steps, 0, g=W.G, H0=W.H0, host_steps=False, **kw)
    c, sc, gc = _run(N, k, init, steps, 0, g=W.G, H0=W.H0, host_steps=True, **kw)
    for x, y in zip(a, c):
        assert np.array_equal(x, y), name
    for f in ("krylov_iterations", "last_krylov_iterations", "last_rel_residual", "steps"):
        assert sa[f] == sc[f], f
    assert ga == gc and sa["kernel_launches"] > 4 * sa["krylov_iterations"] > 0


@pytest.mark.parametrize("N,k,boundary,kw", [
    (8, 2, "periodic", {}), (20, 5, "wall", {}), (33, 3, "periodic", {}), (24, 3, "periodic", dict(krylov_restart=1)),
    (32, 2, "periodic", ASSEMBLED), (47, 4, "periodic", ASSEMBLED), (91, 3, "periodic", ASSEMBLED),
    (16, 7, "wall", ASSEMBLED), (40, 3, "periodic", dict(ASSEMBLED, krylov_ortho=1)),
    (15, 1, "periodic", dict(precision="mixed"))])
def test_paths_and_grids_agree(N, k, boundary, kw):
    init = _large(N, k, boundary)
    tol = 1e-6 if kw.get("precision") == "mixed" else 1e-9
    want, st, _ = _run(N, k, init, 6, 0, boundary=boundary, **kw)
    for blocks in (-1, 1, 7, 32, 1000):
        got, sg, _ = _run(N, k, init, 6, blocks, boundary=boundary, **kw)
        for a, c in zip(got, want):
            assert np.linalg.norm(a - c) <= tol * np.linalg.norm(c)
        assert sg["last_rel_residual"] <= (1e-9 if kw.get("precision") == "mixed" else 1e-12)


def test_the_path_may_change_between_steps():
    """Back and forth on one handle: the other path's basis lies where the exchanged words do."""
    N, k = 24, 3
    init = _large(N, k)
    for kw in ({}, ASSEMBLED):
        want, _, _ = _run(N, k, init, 8, -1, **kw)
        with hd.Sim(N, k, init[4], bottom=init[3], **kw) as s:
            s.set_state(*init[:3])
            for blocks in (-1, 0, 9, 0, -1, -1, 3, 0):
                s.set_solve_blocks(blocks)
                s.step(1)
            got = s.get_state()
        for a, c in zip(got, want):
            assert np.linalg.norm(a - c) <= (1e-6 if kw else 1e-9) * np.linalg.norm(c)
