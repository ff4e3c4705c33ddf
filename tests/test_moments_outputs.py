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


@pytest.mark.parametrize("kind", ["plain", "negated", "zero", "strided"])
def test_init_reads_the_values_of_lazy_views(monkeypatch, kind):
    """The library reads a field's memory: a view whose values are not what its memory holds
    has to be written out first."""
    got = []

    def read(h, rho, *u):
        assert all(c.is_contiguous() and not c.is_neg() for c in u)
        got.append([c.reshape(-1).numpy().copy() for c in u])

    sim = _wrapper(monkeypatch, lbmrv_init_equilibrium_fields=read,
                   lbmrv_init_equilibrium=lambda h, rho, u: read(h, rho, *u))
    base = torch.arange(12.0).reshape(3, 4)
    field = {"plain": base, "negated": torch._neg_view(base),
             "zero": torch._efficientzerotensor((3, 4)),
             "strided": torch.arange(24.0).reshape(3, 8)[:, ::2]}[kind]
    want = {"plain": base, "negated": -base, "zero": 0 * base,
            "strided": 2 * base}[kind].reshape(-1).tolist()
    sim.init_equilibrium(torch.ones(3, 4), field, base)
    assert got[0][0].tolist() == want and got[0][1].tolist() == base.reshape(-1).tolist()
