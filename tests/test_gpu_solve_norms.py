"""The one-launch solve's ||g||, from which its tolerance and the reported residual follow, against the
launch-per-operation path's, on steps whose start is extrapolated (mixed form).

Both square the same FP32 values; there the squares are added in FP64, in the one launch as FP32 pairs.
The sum of n positive terms over at most 12 levels of pair additions, each within 2^-47 of its result, is
within 8.6e-14, its root within 4.3e-14; the FP64 sums add a few 1e-16: 1e-13.  Sizes at which a thread
of the other path has one value (its FP32 chain has then one term)."""
import numpy as np
import pytest

from paper_1711_02751_gb300 import workloads as W

pytestmark = pytest.mark.gpu
hd = pytest.importorskip("paper_1711_02751_gb300.hdgdg")

ASSEMBLED = dict(precision="mixed", local_precision="f32x2", residual_f32x2=True)


@pytest.mark.parametrize("N,k", [(24, 3), (40, 3), (32, 2), (47, 4), (7, 1)])
def test_reported_residuals_agree_between_the_paths(N, k):
    x, y = hd.node_coords(N, k)
    h, hu, hv, b = W.large_state(x, y, seed=11)
    dt = W.advective_dt(x, h, hu, hv, N)
    got = []
    for blocks in (-1, 0):
        with hd.Sim(N, k, dt, bottom=b, **ASSEMBLED) as s:
            s.set_solve_blocks(blocks)
            s.set_state(h, hu, hv)
            rel = []
            for _ in range(4):
                s.step(1)
                rel.append((s.stats()["last_rel_residual"], s.get_state()))
            got.append(rel)
    compared = 0
    for (a, sa), (c, sc) in zip(*got):
        if not all(np.array_equal(p, q) for p, q in zip(sa, sc)):
            break                                  # another trajectory: nothing left to compare
        assert abs(a / c - 1.0) <= 1e-13
        compared += 1
    assert compared >= 2                           # at least one extrapolated start
