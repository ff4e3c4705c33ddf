"""How a call's steps are split into launches: planning it and reading it."""
import time

import pytest

pytestmark = pytest.mark.gpu

S = [0, 0, 0, 1.4, 1.9, 1.7, 1.2, 1.1, 1.3]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _host_us_per_call(torch, sim, calls, repeats=200):
    """Least host time of a call over a few series (the launches queue up behind a kernel)."""
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(repeats):
            for call in calls:
                call()
        best = min(best, time.perf_counter() - t)
    torch.cuda.synchronize()
    return best / (repeats * len(calls)) * 1e6


def test_changing_step_counts_are_not_planned_again():
    """Calls of 5 and 6 steps in turn, and of 5 steps with a new amplitude each, take the host
    no longer than twice the launches of equal calls (one of 5 steps, two of 3)."""
    import torch

    from paper_1312_3297_gb300 import D2Q9

    sim = D2Q9(64, 64, S, mode="prescribed")
    sim.set_utilde(None, 0.03, 0.0)
    one = torch.ones(64, 64, device="cuda")
    sim.init_equilibrium(one, 0 * one, 0 * one)
    five, six = (lambda: sim.step(5)), (lambda: sim.step(6))
    amp = iter(range(10 ** 9))
    new = lambda: sim.set_utilde(None, 0.03 + 1e-9 * next(amp), 0.0)  # noqa: E731
    for f in (five, six, new):
        f()
    base = _host_us_per_call(torch, sim, [five]) + _host_us_per_call(torch, sim, [six])
    assert _host_us_per_call(torch, sim, [five, six]) <= 2.0 * base / 2
    assert _host_us_per_call(torch, sim, [new, five]) <= 2.0 * (
        _host_us_per_call(torch, sim, [five]) + _host_us_per_call(torch, sim, [new])) / 2
    sim.close()
