"""Requests share the device: every handle the serving loop steps has its trace solves bounded to a fixed
share of the SMs before its first step, the same for lone runs, requests and batches (no GPU: a stand-in
for the library's handle records the calls)."""
import numpy as np
import pytest

hd = pytest.importorskip("paper_1711_02751_gb300.hdgdg")
from paper_1711_02751_gb300 import serving  # noqa: E402


class Handle:
    made = []

    def __init__(self, N, k, dt, batch=1, **kw):
        self.shape, self.calls = (batch * N * N, (k + 1) ** 2), []
        Handle.made.append(self)

    def __enter__(self):
        return self

    def __exit__(self, *a):
        return False

    def set_solve_blocks(self, n):
        self.calls.append(("blocks", n))

    def set_state(self, h, hu, hv):
        self.calls.append(("state",))

    def step(self, n):
        self.calls.append(("step", n))

    def get_state(self):
        return tuple(np.zeros(self.shape) for _ in range(3))


def test_served_handles_take_a_fixed_share_of_the_sms(monkeypatch):
    monkeypatch.setattr(serving.hd, "Sim", Handle)
    Handle.made.clear()
    reqs = serving.ensemble_requests(n=12, sides=(4, 6), degrees=(2, 3), steps=5)
    assert serving.Server(1 << 34).serve(serving.batch_requests(reqs[:8]))["completed"] == 8
    assert serving.Server(1 << 34).serve(reqs[8:])["completed"] == 4
    serving.run_one(reqs[0])
    limits = set()
    for s in Handle.made:
        first = s.calls.index(next(c for c in s.calls if c[0] == "step"))
        limits |= {c[1] for c in s.calls[:first] if c[0] == "blocks"}
        assert any(c[0] == "blocks" for c in s.calls[:first])
    assert len(limits) == 1 and 0 < limits.pop() <= 152 // 3
