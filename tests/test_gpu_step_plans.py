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


@pytest.mark.parametrize("storage,lanes", [("fp32", 512), ("fp16", 1024)])
@pytest.mark.parametrize("blocks,ny", [(4096, 1), (4097, 1), (4096, 2), (4097, 2), (66000, 2)])
def test_fused_sums_of_very_wide_rows(storage, lanes, blocks, ny):
    """Rows of as many blocks as the step's last block adds, one more, and of more than 256
    middle sums: the separate pass's sums, the same in every run."""
    import numpy as np
    import torch

    from paper_1312_3297_gb300 import D2Q9

    nx = (blocks - 1) * lanes + 8  # the last block holds one or two packs
    sim = D2Q9(nx, ny, S, storage=storage)
    gen = torch.Generator(device="cuda").manual_seed(blocks)
    r = [torch.randn(ny, nx, generator=gen, device="cuda") for _ in range(3)]
    runs = []
    for _ in range(2):
        sim.init_equilibrium(1.0 + 0.01 * r[0], 0.05 + 0.01 * r[1], 0.02 + 0.01 * r[2])
        runs.append([sim.step_conserved(1) for _ in range(2)])
    # the tolerance of the other fused sums: FP32 runs of 32 nodes, then FP64
    np.testing.assert_allclose(runs[0][1][:4], sim.conserved3()[:4], rtol=1e-12,
                               atol=1e-9 * nx * ny)
    assert runs[0] == runs[1] and runs[0][1][4] == 0.0
    sim.close()
