"""Each form of the D2Q9 step (three steps per pass over memory, several per launch on tiles of
both widths), forced and seen to be the one that runs, against single-step launches: the same
states bit for bit, in the same buffer, over every relaxation that the one-step kernels use
(storage, relative velocity, basis, pack width)."""
import pytest

pytestmark = pytest.mark.gpu

S = [0, 0, 0, 1.4, 1.9, 1.7, 1.2, 1.1, 1.3]
EVERY = [pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"]),
         pytest.mark.parametrize("mode", ["zero", "fluid", "prescribed", "field"]),
         pytest.mark.parametrize("lattice", ["D2Q9", "D2Q9Cascaded"])]


def every(test):
    for mark in EVERY:
        test = mark(test)
    return test


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _pair(lattice, nx, ny, mode, storage, form):
    import torch

    import paper_1312_3297_gb300 as pkg

    gen = torch.Generator(device="cuda").manual_seed(nx + ny)
    r = [torch.randn(ny, nx, generator=gen, device="cuda") for _ in range(3)]
    ut0 = torch.randn(2, ny, nx, generator=gen, device="cuda") if mode == "field" else None
    sims = []
    for f in ("single", form):
        sim = getattr(pkg, lattice)(nx, ny, S, mode="prescribed" if mode == "field" else mode,
                                    storage=storage)
        if mode in ("prescribed", "field"):
            sim.set_utilde(ut0, 0.05, 9.0)
        sim.init_equilibrium(1.0 + 0.01 * r[0], 0.05 + 0.01 * r[1], 0.02 + 0.01 * r[2])
        sim.set_step_form(f)
        sims.append(sim)
    return sims


def _same(one, many, n):
    import torch

    one.step(n)
    many.step(n)
    assert one.time == many.time
    assert torch.equal(one.state().view(torch.uint8), many.state().view(torch.uint8)), n
    assert (one.state_ptr() == one._bufs[0].data_ptr()) == (
        many.state_ptr() == many._bufs[0].data_ptr())


# one pack; as few rows as the rows that a strip carries and recomputes, or fewer (the march laps
# the lattice); full and partial strips; 16-bit rows that 8-node packs do not divide
MARCH_TINY = [(4, 1), (4, 2), (8, 3), (12, 4), (64, 64), (128, 1), (132, 2), (124, 5), (480, 7),
              (484, 6), (248, 11)]
MARCH = [(4, 90001), (128, 2500), (132, 2500), (1800, 2003), (1804, 2001), (1796, 2003),
         (13108, 28), (2052, 1801)]


@every
def test_march(lattice, mode, storage):
    for sizes, counts in ((MARCH_TINY, (3, 4, 7, 25)), (MARCH, (3, 7, 26))):
        for nx, ny in sizes:
            if (mode, lattice) == ("field", "D2Q9Cascaded") and storage != "fp32" and nx % 8:
                continue  # refused: see below
            one, many = _pair(lattice, nx, ny, mode, storage, "march")
            for n in counts:
                assert one.step_plan(n) == ("single", n, 1, 0)
                assert many.step_plan(n) == ("march", n // 3 + n % 3, 3, 0)
                _same(one, many, n)


# per pack width of the one-step kernels: small and large enough for arrays of 32 and of 64 nodes
TILE = {1: [(1, 1), (1, 9), (9, 1), (63, 41), (33, 130), (901, 700)],
        2: [(2, 3), (2, 1), (130, 77), (902, 700)],
        4: [(36, 300), (300, 36), (900, 701)],
        8: [(64, 64), (8, 40), (520, 260), (904, 700)]}


@every
@pytest.mark.parametrize("width", [1, 2, 4, 8])
def test_tile(lattice, mode, storage, width):
    seen = set()
    for nx, ny in TILE[width]:
        one, many = _pair(lattice, nx, ny, mode, storage, "tile")
        for n in (5, 6, 7, 12, 25) if nx * ny < 100000 else (5, 7, 8):
            form, launches, longest, rx = many.step_plan(n)
            assert form == "tile" and launches < n and (launches - n) % 2 == 0
            assert longest == -(-n // launches)
            seen.add(rx)
            _same(one, many, n)
    assert seen == {32, 64}


def test_refused_forms():
    import torch

    from paper_1312_3297_gb300 import D2Q9, D2Q9Cascaded, D3Q19
    from paper_1312_3297_gb300 import binding as B

    def refused(sim, form):
        with pytest.raises(B.LbmrvError, match="LBMRV_E_(INVAL|UNSUPPORTED)"):
            B.lbmrv_set_step_form(sim.h, form)
        assert sim.step_plan(1) == ("single", 1, 1, 0)

    sim = D2Q9(66, 8, S)
    refused(sim, B.LBMRV_FORM_MARCH)  # rows of whole 4-node packs only
    refused(sim, 4)
    refused(sim, -1)
    sim = D2Q9Cascaded(68, 8, S, mode="prescribed", storage="fp16")
    sim.set_utilde(torch.zeros(2, 8, 68, device="cuda"), 0.1, 0.0)
    refused(sim, B.LBMRV_FORM_MARCH)  # Geier's 4-node 16-bit packs of a stored field
    sim = D3Q19(8, 8, 8, [0, 0, 0, 0] + [1.2] * 15)
    refused(sim, B.LBMRV_FORM_MARCH)
    refused(sim, B.LBMRV_FORM_TILE)
    assert sim.step_plan(5) == ("single", 5, 1, 0)


def test_plan_follows_the_width_and_the_count():
    from paper_1312_3297_gb300 import D2Q9

    sim = D2Q9(64, 64, S)
    assert sim.step_plan(0) == ("single", 0, 0, 0)
    assert sim.step_plan(2) == ("single", 2, 1, 0)
    assert sim.step_plan(20)[0] == "tile"
    sim.set_kernel_width(4)
    assert sim.step_plan(20) == ("single", 20, 1, 0)


# lattices whose states fit L2 or nearly do, where the forms' times cross
CROSSING = [("D2Q9Cascaded", 1560, 656, "fp32", "field", 7),
            ("D2Q9Cascaded", 928, 1528, "fp32", "prescribed", 7),
            ("D2Q9Cascaded", 352, 2369, "fp32", "zero", 10),
            ("D2Q9Cascaded", 2024, 734, "fp32", "prescribed", 10),
            ("D2Q9", 160, 1136, "fp16", "fluid", 4),
            ("D2Q9", 528, 1504, "fp32", "prescribed", 4),
            ("D2Q9", 352, 1464, "fp32", "field", 100)]


@pytest.mark.parametrize("lattice,nx,ny,storage,mode,n", CROSSING)
def test_the_chosen_form_is_not_slower_than_single_steps(lattice, nx, ny, storage, mode, n):
    """Calls of n steps back to back, in turn with single steps, best of several series; the
    margin is for what is left of the models' error (two series differ by under 2 %)."""
    import torch

    one, auto = _pair(lattice, nx, ny, mode, storage, "auto")
    calls = max(4, 200 // n)
    best = {}
    for _ in range(6):
        for sim in (one, auto):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            sim.step(n)
            torch.cuda.synchronize()
            torch.cuda._sleep(200000)
            a.record(sim.stream)
            for _ in range(calls):
                sim.step(n)
            b.record(sim.stream)
            b.synchronize()
            best[sim] = min(best.get(sim, float("inf")), a.elapsed_time(b))
    assert best[auto] <= 1.15 * best[one]
