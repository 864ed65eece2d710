"""Explicit steps queued in one call against the same steps called one at a time: bit for bit, past
the 64 steps queued before the host waits, and where a step turns non-finite the state, the time and
the step count are those of the last finite step."""
import numpy as np
import pytest

from paper_1711_02751_gb300 import workloads as W

pytestmark = pytest.mark.gpu
hd = pytest.importorskip("paper_1711_02751_gb300.hdgdg")

V = W.VORTEX
VORTEX = dict(boundary="vortex", x0=-2.0, length=4.0, g=V["g"], H0=V["H_inf"],
              bc_params=(V["beta"], V["u_inf"], V["v_inf"], V["xc"], V["yc"]))


def _run(calls, N, k, scheme, courant, kw):
    """Status, steps done and state after the calls, stopping at the first that fails."""
    rng = np.random.default_rng(N + k)
    nn = (N * N, (k + 1) ** 2)
    dt = courant * kw.get("length", 1.0) / (N * (2 * k + 1))
    h, hu, hv = 1.0 + 0.01 * rng.standard_normal(nn), 0.01 * rng.standard_normal(nn), 0.01 * rng.standard_normal(nn)
    with hd.Sim(N, k, dt, np.zeros(nn), scheme=scheme, **kw) as s:
        s.set_state(h, hu, hv)
        status = 0
        try:
            for c in calls:
                s.step(c)
        except hd.HdgdgError as ex:
            status = ex.status
        return status, s.stats()["steps"], s.get_state()


@pytest.mark.parametrize("scheme", ["rk2", "rk3"])
@pytest.mark.parametrize("N,k,courant,kw", [(5, 1, 0.2, {}), (4, 8, 0.2, {}), (6, 3, 0.2, dict(boundary="wall")),
                                            (3, 4, 0.05, VORTEX), (4, 3, 30.0, {})])
def test_queued_steps_equal_single_steps(N, k, scheme, courant, kw):
    n = 131
    one = _run([1] * n, N, k, scheme, courant, kw)
    many = _run([n], N, k, scheme, courant, kw)
    assert one[:2] == many[:2]
    if courant > 1.0:
        assert one[0] == hd.ENONFINITE
    for a, b in zip(one[2], many[2]):
        assert np.isfinite(a).all() and np.array_equal(a, b)
