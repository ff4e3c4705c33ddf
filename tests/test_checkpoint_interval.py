"""The default checkpoint interval of a rollout (host logic, no GPU)."""
import math
import types

import pytest

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 2, 9, 200, 2000])
@pytest.mark.parametrize("total_gb", [0.1, 16.0, 280.0])
def test_interval_is_the_shortest_within_the_share(monkeypatch, n, total_gb):
    from paper_1312_3297_gb300 import autograd

    state = 36 << 20  # bytes of one state at 1024^2
    sim = types.SimpleNamespace(
        device="cuda:0",
        adjoint_workspace_bytes=lambda n, seg: (-(-n // seg) + seg - 1 + 2) * state)
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d: types.SimpleNamespace(total_memory=total_gb * 2 ** 30))
    seg = autograd.checkpoint_interval(sim, n)
    budget = autograd.CHECKPOINT_SHARE * total_gb * 2 ** 30
    longest = max(1, math.ceil(math.sqrt(n)))
    assert 1 <= seg <= longest
    if seg < longest:
        assert sim.adjoint_workspace_bytes(n, seg) <= budget
    if seg > 1:
        assert sim.adjoint_workspace_bytes(n, seg - 1) > budget
