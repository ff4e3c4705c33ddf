"""Results read through the handles' shared pages of mapped host memory: more handles than a page
has slots, given back out of order, and from several threads."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

S = [0, 0, 0, 1.4, 1.9, 1.9, 1.2, 1.2, 1.4]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _sim(k):
    import torch

    from paper_1312_3297_gb300 import D2Q9

    sim = D2Q9(8, 4, S)
    rho = torch.full((4, 8), 1.0 + k / 256, device="cuda")  # exact in FP32
    sim.init_equilibrium(rho, torch.zeros_like(rho), torch.zeros_like(rho))
    return sim


def _check(sim, k):
    assert sim.conserved()[0] == pytest.approx(32 * (1.0 + k / 256), rel=1e-6)


@pytest.mark.parametrize("count", [1, 64, 65, 150])
def test_many_handles(count):
    sims = {k: _sim(k) for k in range(count)}
    for k in np.random.default_rng(count).permutation(count)[: count // 2]:
        sims.pop(int(k)).close()
    for k in range(count, count + count // 3):
        sims[k] = _sim(k)
    for k, sim in sims.items():
        _check(sim, k)
    for sim in sims.values():
        sim.close()


def test_threads():
    failures = []

    def work(base):
        try:
            for k in range(base, base + 25):
                sim = _sim(k)
                sim.step(3)
                _check(sim, k)
                sim.close()
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            failures.append(e)

    threads = [threading.Thread(target=work, args=(25 * i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures
