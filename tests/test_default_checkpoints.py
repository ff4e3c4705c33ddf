"""Memory of rollouts that name no checkpoint interval."""
import gc
import math
import types

import pytest

torch = pytest.importorskip("torch")

STATE = 36 << 20  # bytes of one state at 1024^2
N = 200


class _Sim:
    """Workspace sizes of a 1024^2 lattice; the workspaces themselves are small."""

    device = torch.device("cuda", 0)

    def __init__(self, device_memory):
        self.memory = device_memory

    def adjoint_workspace_bytes(self, n, seg):
        return (-(-n // seg) + seg - 1 + 2) * STATE

    def adjoint_workspace(self, n, seg):
        size = self.adjoint_workspace_bytes(n, seg)
        if size > self.memory.free:
            raise torch.cuda.OutOfMemoryError("no room")
        ws = torch.empty(1)
        ws.memory = self.memory.take(size)
        return ws


class _Memory:
    def __init__(self, free):
        self.free, self.told = free, None

    def take(self, size):
        memory = self

        class Lease:
            def __init__(self):
                memory.free -= size

            def __del__(self):
                memory.free += size

        return Lease()


@pytest.fixture
def autograd(monkeypatch):
    from paper_1312_3297_gb300 import autograd as module

    gc.collect()
    monkeypatch.setattr(module, "_extra", {})
    monkeypatch.setattr(module, "_seen", {})
    return module


TOTAL = 280 << 30


def _use(monkeypatch, memory):
    def info(index):
        return (memory.told if memory.told is not None else memory.free), TOTAL

    monkeypatch.setattr(torch.cuda, "cudart", lambda: types.SimpleNamespace(cudaMemGetInfo=info))
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d: types.SimpleNamespace(total_memory=TOTAL))
    return _Sim(memory)


LONGEST = math.ceil(math.sqrt(N))


def test_many_live_rollouts_together_stay_within_the_share(monkeypatch, autograd):
    """As many rollouts as fit with sqrt(n) checkpoints and an eighth of the memory spare: every
    one is served, and together they hold no more than that eighth beyond what sqrt(n)
    checkpoints hold."""
    memory = _Memory(TOTAL)
    sim = _use(monkeypatch, memory)
    least = sim.adjoint_workspace_bytes(N, LONGEST)
    count = int(TOTAL * (1 - autograd.LIVE_SHARE) / least)
    live = []
    for k in range(count):
        live.append(autograd.default_workspace(sim, N))
        assert TOTAL - memory.free <= (k + 1) * least + autograd.LIVE_SHARE * TOTAL
    assert live[2][0] == 1 and live[-1][0] > 1
    del live
    gc.collect()
    assert memory.free == TOTAL and autograd._extra == {sim.device: 0}
    assert autograd.default_workspace(sim, N)[0] == 1  # given back


def test_the_free_memory_is_looked_at_again(monkeypatch, autograd):
    """Memory that others took a moment ago is not counted as free, and an allocation that
    fails makes the next rollout look at once."""
    sim = _use(monkeypatch, _Memory(TOTAL))
    clock = [100.0]
    monkeypatch.setattr(autograd.time, "monotonic", lambda: clock[0])
    least = sim.adjoint_workspace_bytes(N, LONGEST)
    assert autograd.default_workspace(sim, N)[0] == 1
    sim.memory.free = least + (64 << 20)  # taken by others
    seg, ws = autograd.default_workspace(sim, N)
    assert sim.adjoint_workspace_bytes(N, seg) == least  # the failed allocation's fallback
    del ws
    sim.memory.free = 8 << 30
    seg, ws = autograd.default_workspace(sim, N)  # fits, but would leave nothing spare
    assert sim.adjoint_workspace_bytes(N, seg) < least + autograd.LIVE_SHARE * (8 << 30)
    del ws
    sim.memory.free = TOTAL
    clock[0] += 2 * autograd.LOOK_SECONDS
    assert autograd.default_workspace(sim, N)[0] == 1


def test_one_rollout_stays_within_its_share(monkeypatch, autograd):
    sim = _use(monkeypatch, _Memory(TOTAL))
    n = 4000
    seg, ws = autograd.default_workspace(sim, n)
    assert 1 < seg < math.ceil(math.sqrt(n))
    assert sim.adjoint_workspace_bytes(n, seg) <= autograd.CHECKPOINT_SHARE * TOTAL
    assert sim.adjoint_workspace_bytes(n, seg - 1) > autograd.CHECKPOINT_SHARE * TOTAL


def test_small_workspaces_need_no_look_at_the_memory(monkeypatch, autograd):
    sim = _use(monkeypatch, _Memory(TOTAL))
    monkeypatch.setattr(torch.cuda, "cudart", None)
    assert autograd.default_workspace(sim, 9)[0] == 1


def test_little_free_memory_means_least_memory(monkeypatch, autograd):
    sim = _use(monkeypatch, _Memory(0))
    least = sim.adjoint_workspace_bytes(N, LONGEST)
    sim.memory.free = least + (64 << 20)
    seg, ws = autograd.default_workspace(sim, N)
    assert sim.adjoint_workspace_bytes(N, seg) == least


def test_a_failed_allocation_falls_back(monkeypatch, autograd):
    """The driver reports free memory that the allocation then does not get."""
    memory = _Memory(2 << 30)
    memory.told = TOTAL
    sim = _use(monkeypatch, memory)
    seg, ws = autograd.default_workspace(sim, N)
    assert seg == LONGEST and autograd._extra == {sim.device: 0}


def test_one_step(monkeypatch, autograd):
    sim = _use(monkeypatch, _Memory(1 << 30))
    assert autograd.default_workspace(sim, 1)[0] == 1 and autograd._extra == {}


def test_invalid_windows_are_refused(monkeypatch, autograd):
    sim = _use(monkeypatch, _Memory(TOTAL))
    monkeypatch.setattr(_Sim, "adjoint_workspace_bytes", lambda self, n, seg: -1)

    def refuse(self, n, seg):
        raise ValueError("invalid adjoint window")

    monkeypatch.setattr(_Sim, "adjoint_workspace", refuse)
    with pytest.raises(ValueError):
        autograd.default_workspace(sim, N)
    assert autograd._extra == {sim.device: 0}


@pytest.mark.gpu
@pytest.mark.parametrize("fails", [False, True])
def test_default_gradient_equals_that_of_a_given_interval(fails):
    """The gradient of a rollout that names no interval, with and without room for its dense
    checkpoints, equals that with 7 steps between checkpoints bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1312_3297_gb300 import D2Q9
    from paper_1312_3297_gb300.autograd import Rollout

    nx, ny, steps = 96, 64, 50
    gen = torch.Generator(device="cuda").manual_seed(3)
    start = 0.05 * torch.randn(2, ny, nx, generator=gen, device="cuda")
    grads, segs = [], []
    for seg in (7, 0):
        sim = D2Q9(nx, ny, [0, 0, 0, 1.4, 1.9, 1.9, 1.2, 1.2, 1.4])
        make = sim.adjoint_workspace

        def workspace(n, s, make=make, seg=seg):
            segs.append(s)
            if fails and seg == 0 and s == 1:
                raise torch.cuda.OutOfMemoryError("no room")
            return make(n, s)

        sim.adjoint_workspace = workspace
        u0 = start.clone().requires_grad_()
        s_nu = torch.tensor(1.9, dtype=torch.float64, requires_grad=True)
        rho, u = Rollout.apply(u0, s_nu, torch.tensor(0.0), sim, steps, seg, None)
        (rho * (u * u).sum(0)).sum().backward()
        grads.append((u0.grad, s_nu.grad))
        sim.close()
    assert segs == ([7, 1, math.ceil(math.sqrt(steps))] if fails else [7, 1])
    assert torch.equal(grads[0][0], grads[1][0]) and torch.equal(grads[0][1], grads[1][1])
