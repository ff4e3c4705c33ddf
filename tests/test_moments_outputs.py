"""What ``moments`` and ``init_equilibrium`` hand over and take (host logic, no GPU)."""
import types

import pytest

torch = pytest.importorskip("torch")


def _wrapper(monkeypatch, **entries):
    """A D2Q9 on the CPU whose library entry points are replaced."""
    from paper_1312_3297_gb300 import simulation

    sim = object.__new__(simulation.D2Q9)
    sim.device, sim.shape, sim.n, sim.h = torch.device("cpu"), (3, 4), 12, None
    monkeypatch.setattr(sim, "_on_current_stream", lambda: True)
    monkeypatch.setattr(sim, "_sync_in", lambda: None)
    monkeypatch.setattr(sim, "_sync_out", lambda: None)
    monkeypatch.setattr(simulation, "B", types.SimpleNamespace(**entries))
    return sim


@pytest.mark.parametrize("k", [0, 1, 2])
def test_a_field_can_be_changed_in_place_under_autograd(monkeypatch, k):
    sim = _wrapper(monkeypatch, lbmrv_moments=lambda h, rho, u: (rho.fill_(1.0), u.fill_(2.0)))
    p = torch.full((3, 4), 0.5, requires_grad=True)
    field = sim.moments()[k]
    field += p
    (3.0 * field).sum().backward()
    assert torch.equal(p.grad, torch.full((3, 4), 3.0))
