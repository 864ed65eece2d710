"""A wait of the one-launch trace solve that runs out (a contribution that never comes; every wait is bounded
to about a second): the launch ends by itself, the call returns ECUDA and the device stays usable."""
import numpy as np
import pytest

from paper_1711_02751_gb300 import workloads as W

pytestmark = pytest.mark.gpu
hd = pytest.importorskip("paper_1711_02751_gb300.hdgdg")

FORMS = {"fp64": {}, "mixed": dict(precision="mixed", local_precision="f32x2", residual_f32x2=True)}


def _state(N, k):
    x, y = hd.node_coords(N, k)
    h, hu, hv, b = W.large_state(x, y, seed=7)
    return h, hu, hv, b, W.advective_dt(x, h, hu, hv, N)


@pytest.mark.parametrize("host_steps", [False, True])
@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_a_lost_contribution_ends_the_step_with_an_error(form, host_steps):
    h, hu, hv, b, dt = _state(24, 3)
    with hd.Sim(24, 3, dt, bottom=b, host_steps=host_steps, **FORMS[form]) as s:
        s.set_state(h, hu, hv)
        s.step(2)
        before = s.get_state()
        s.lose_contribution()
        with pytest.raises(hd.HdgdgError) as ex:
            s.step(1)
        assert ex.value.status == hd.ECUDA and "wait" in str(ex.value)
        assert s.stats()["steps"] == 2
        for a, c in zip(before, s.get_state()):
            assert np.array_equal(a, c)
    with hd.Sim(24, 3, dt, bottom=b, host_steps=host_steps, **FORMS[form]) as s:
        s.set_state(h, hu, hv)
        s.step(2)
        for a, c in zip(before, s.get_state()):
            assert np.array_equal(a, c)


def test_only_one_launch_solves_have_such_waits():
    h, hu, hv, b, dt = _state(8, 2)
    with hd.Sim(8, 2, dt, bottom=b, precision="mixed", local_precision="f32x2", trace_operator=1) as s:
        with pytest.raises(hd.HdgdgError) as ex:
            s.lose_contribution()
        assert ex.value.status == hd.EINVAL


@pytest.mark.parametrize("host_steps", [False, True])
@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_the_handle_goes_on_after_a_lost_contribution(form, host_steps):
    """The exchange's numbers and words start afresh: the steps after the failed one are those of a handle
    that lost nothing, bit for bit, again and again, and so is a stage solve."""
    h, hu, hv, b, dt = _state(24, 3)
    with hd.Sim(24, 3, dt, bottom=b, host_steps=host_steps, **FORMS[form]) as s, \
            hd.Sim(24, 3, dt, bottom=b, host_steps=host_steps, **FORMS[form]) as ref:
        s.set_state(h, hu, hv)
        s.step(3)
        for steps, scale in ((1, 1.0), (6, 0.5)):
            for sim in (s, ref):
                sim.set_state(h, scale * hu, scale * hv)
            s.lose_contribution()
            with pytest.raises(hd.HdgdgError) as ex:
                s.step(1)
            assert ex.value.status == hd.ECUDA
            s.step(steps)
            ref.step(steps)
            for a, c in zip(ref.get_state(), s.get_state()):
                assert np.array_equal(a, c)
        R1 = np.random.default_rng(3).standard_normal((3, 24 * 24, 16))
        want = ref.stage_solve(R1)[1]
        s.lose_contribution()
        with pytest.raises(hd.HdgdgError):
            s.stage_solve(R1)
        assert np.array_equal(s.stage_solve(R1)[1], want)


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_the_timers_leave_a_failed_launch_out(form):
    """With the kernel-class timers on, the launch that gave up after most of a second is in no class, and
    the steps after it are timed."""
    h, hu, hv, b, dt = _state(24, 3)
    with hd.Sim(24, 3, dt, bottom=b, **FORMS[form]) as s:
        s.set_state(h, hu, hv)
        s.set_kernel_timing(True)
        s.step(2)
        s.lose_contribution()
        with pytest.raises(hd.HdgdgError):
            s.step(1)
        s.step(2)
        times = s.kernel_times()
    assert all(times[c][0] > 0.0 for c in ("spmv", "ortho", "residual", "guess", "precond"))
    assert sum(ms for ms, _ in times.values()) < 100.0
