"""The trace solve as one cooperative launch (small and mid-size systems on the assembled matrix):
its solution against the library's own operator and right-hand side, which run other kernels.

stage_solve gives qhat for a random R1; S qhat (trace_apply) must equal g (condense_rhs) to the solve's
stop test: 1e-9 ||g|| in the mixed form (its residual is FP64-class, 1e-13), the FP64 floor of 1e-12
||g|| plus the rounding of both products (1e-14 of |S||x|, below 1e-11 ||g|| on these meshes) in the
FP64 form.  Sizes: fewer edges than one block takes, a ragged last block, every split of a row's
columns (k = 1..8), restart lengths 1 and 31, absent sides and prescribed traces, an FP32 basis that
all but fills shared memory (128^2, k = 3) and the first size past it, which keeps the
launch-per-operation path; there restart lengths that cover every width of its column reductions."""
import numpy as np
import pytest

from paper_1711_02751_gb300 import workloads as W

pytestmark = pytest.mark.gpu
hd = pytest.importorskip("paper_1711_02751_gb300.hdgdg")

FAST = dict(precision="mixed", local_precision="f32x2", residual_f32x2=True)
MIXED = dict(precision="mixed")
MF = dict(precision="mixed", local_precision="f32x2", trace_operator=1)
V = W.VORTEX
VORTEX = dict(boundary="vortex", x0=-2.0, length=4.0, g=V["g"], H0=V["H_inf"],
              bc_params=(V["beta"], V["u_inf"], V["v_inf"], V["xc"], V["yc"]))


@pytest.mark.parametrize("N,k,kw", [
    (2, 1, {}), (3, 8, {}), (8, 2, dict(krylov_restart=1)), (16, 3, dict(krylov_restart=31)),
    (5, 4, dict(boundary="wall")), (6, 5, VORTEX), (9, 6, {}), (7, 7, {}), (96, 3, {}),
    (2, 2, FAST), (33, 2, FAST), (12, 1, FAST), (47, 4, FAST), (20, 5, MIXED), (11, 6, FAST), (13, 7, FAST),
    (9, 8, FAST), (6, 3, dict(FAST, boundary="wall")), (6, 4, dict(FAST, **VORTEX)),
    (24, 3, dict(FAST, krylov_restart=1)), (24, 2, dict(MIXED, krylov_restart=31)),
    (40, 3, dict(FAST, krylov_ortho=1)), (128, 3, FAST), (160, 3, FAST),
    # the launch-per-operation path: reductions of up to 32 columns at once, and the FP64 form's
    (24, 3, dict(MF, krylov_restart=31)), (15, 2, dict(MF, krylov_restart=3)), (120, 3, dict(krylov_restart=31))])
def test_solution_satisfies_the_trace_system(N, k, kw):
    rng = np.random.default_rng(N * 10 + k)
    kw = dict(kw)
    nn = (N * N, (k + 1) ** 2)
    x, y = hd.node_coords(N, k, boundary=kw.get("boundary", "periodic"), x0=kw.get("x0", 0.0),
                          length=kw.get("length", 1.0))
    b = np.zeros(nn) if "bc_params" in kw else 0.1 * np.sin(2 * np.pi * x) * np.sin(2 * np.pi * y)
    dt = 0.5 * kw.get("length", 1.0) / N / (2 * k + 1)
    with hd.Sim(N, k, dt, bottom=b, **kw) as s:
        R1 = rng.standard_normal((3,) + nn)
        g = s.condense_rhs(R1)
        _, qhat, its = s.stage_solve(R1)
        res = np.linalg.norm(s.trace_apply(qhat) - g)
        _, again, its2 = s.stage_solve(R1)
    assert its > 0 and its2 == its and np.array_equal(qhat, again)
    assert res <= (1.01e-9 if kw.get("precision") == "mixed" else 1e-11) * np.linalg.norm(g)


def test_streamed_product_past_the_one_launch_size():
    """spmv_kernel chooses the product of the launch-per-operation path: identical steps."""
    N, k = 160, 3
    x, y = hd.node_coords(N, k)
    h, hu, hv, b = W.large_state(x, y, seed=11)
    outs = []
    for kernel in (0, 1):
        with hd.Sim(N, k, W.advective_dt(x, h, hu, hv, N), bottom=b, precision="mixed", spmv_kernel=kernel) as s:
            s.set_state(h, hu, hv)
            s.step(2)
            outs.append(s.get_state())
    for p, q in zip(*outs):
        assert np.array_equal(p, q)


def test_handles_of_different_sizes_in_threads():
    """Handles of one degree and different shared-memory needs created and stepped from eight threads:
    every step succeeds and gives the lone run's state bit for bit."""
    from concurrent.futures import ThreadPoolExecutor

    def run(N):
        nn = (N * N, 9)
        x, y = hd.node_coords(N, 2)
        h = 1.0 + 0.01 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
        with hd.Sim(N, 2, 0.2 / N, np.zeros(nn), **MIXED) as s:
            s.set_state(h, np.zeros(nn), np.zeros(nn))
            s.step(3)
            return np.concatenate([np.ravel(f) for f in s.get_state()])

    sizes = [4, 24, 48, 64]
    lone = {N: run(N) for N in sizes}
    order = sizes * 16
    with ThreadPoolExecutor(8) as pool:
        for N, got in zip(order, pool.map(run, order)):
            assert np.array_equal(got, lone[N])
