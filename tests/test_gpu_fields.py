"""Initial fields: the mean-flow sums against exactly rounded sums, and the equilibrium and the
moments with vector and with single-node accesses (node counts and buffers that four-node packs
do not suit)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

S2 = [0, 0, 0, 1.4, 1.9, 1.9, 1.2, 1.2, 1.4]
S3 = [0, 0, 0, 0, 1.2] + [1.7] * 5 + [1.9] * 6 + [1.4] * 3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _fields(dims, seed, scale=1.0, constant=False):
    rng = np.random.default_rng(seed)
    d = 3 if len(dims) == 3 else 2
    n = int(np.prod(dims))
    rho = np.full(n, 1.1) if constant else 1.0 + 0.1 * rng.standard_normal(n)
    u = np.full((d, n), 0.05) if constant else 0.05 + 0.01 * rng.standard_normal((d, n))
    return (scale * rho).astype(np.float32), u.astype(np.float32)


def _sim(dims, storage="fp32"):
    from paper_1312_3297_gb300 import D2Q9, D3Q19

    return (D3Q19(*dims, S3, storage=storage) if len(dims) == 3 else
            D2Q9(*dims, S2, storage=storage))


# one node, a partial warp, odd counts (single-node loads), whole packs, several blocks, 3D
@pytest.mark.parametrize("dims", [(1, 1), (5, 3), (37, 23), (64, 48), (1000, 701), (1024, 1024),
                                  (7, 5, 3), (64, 40, 24)])
@pytest.mark.parametrize("constant", [False, True])
def test_mean_flow_sums_are_exact_to_fp64_rounding(dims, constant):
    import torch

    from paper_1312_3297_gb300 import binding as B

    sim = _sim(dims)
    # scale 1e9 and 1e-9 take the FP64 kernel
    for scale in (1.0, 1e9, 1e-9):
        rho, u = _fields(dims, 3, scale, constant)
        got = B.lbmrv_flow_sums(sim.h, torch.as_tensor(rho).cuda(), torch.as_tensor(u).cuda())
        r = rho.astype(np.float64)
        ref = [math.fsum(r)] + [math.fsum(r * c) for c in u.astype(np.float64)]
        # products of FP32 values are exact in FP64; at most some 40 FP64 additions in a row,
        # each to 2^-53 of the sum of magnitudes (all terms of one sign but for a few)
        for g, e in zip(got, ref):
            assert abs(g - e) <= 40 * 2.0 ** -53 * max(abs(e), 1e-300)


@pytest.mark.parametrize("dims", [(64, 48), (8, 1), (24, 10, 12)])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_packs_and_single_nodes_give_the_same_state(dims, storage):
    """The same fields from aligned planes (four nodes per access) and from buffers one float
    off (one node per access): populations within the rounding of FP32 (a few 2^-24 of values
    below 1, doubled by the storage rounding of 16 bits), moments of the same state too."""
    import torch

    from paper_1312_3297_gb300 import binding as B

    rho, u = _fields(dims, 5)
    n, d = rho.size, len(u)
    a, b = _sim(dims, storage), _sim(dims, storage)
    t = [torch.as_tensor(c).cuda() for c in (rho, *u)]
    B.lbmrv_init_equilibrium(a.h, t[0], torch.stack(t[1:]))
    off = torch.empty((d + 1, n + 4), device="cuda")
    shifted = [off[k].view(-1)[1:n + 1] for k in range(d + 1)]
    for s, c in zip(shifted, t):
        s.copy_(c)
    B.lbmrv_init_equilibrium_fields(b.h, *shifted)
    assert a.u_ref == pytest.approx(b.u_ref, abs=1e-15)
    x, y = a.state().float(), b.state().float()
    step = {"fp32": 0.0, "fp16": 2.0 ** -10, "bf16": 2.0 ** -7}[storage]
    assert (x - y).abs().max().item() <= 4 * 2.0 ** -24 + step * x.abs().max().item()
    r1, u1 = torch.empty(n, device="cuda"), torch.empty(d * n, device="cuda")
    pad = torch.empty(n + 1, device="cuda")
    r2, u2 = pad[1:], torch.empty(d * n, device="cuda")
    B.lbmrv_moments(a.h, r1, u1)
    B.lbmrv_moments(a.h, r2, u2)
    assert (r1 - r2).abs().max().item() <= 4 * 2.0 ** -24
    assert (u1 - u2).abs().max().item() <= 4 * 2.0 ** -24
    with pytest.raises(B.LbmrvError):
        B.lbmrv_init_equilibrium_fields(b.h, shifted[0], None, shifted[1])
