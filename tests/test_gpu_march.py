"""Several steps per pass over memory (automatic kernel variant) against the same steps taken
one call at a time, each a single-step kernel: the same states bit for bit, in the same buffer.
The single-step kernels are held to the oracle elsewhere."""
import pytest

pytestmark = pytest.mark.gpu

S = [0, 0, 0, 1.4, 1.9, 1.7, 1.2, 1.1, 1.3]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _sim(cls, nx, ny, mode, storage, ut0):
    import torch

    sim = cls(nx, ny, S, mode="prescribed" if mode == "field" else mode, storage=storage)
    if mode in ("prescribed", "field"):
        sim.set_utilde(ut0, 0.05, 9.0)
    gen = torch.Generator(device="cuda").manual_seed(nx + ny)
    r = [torch.randn(ny, nx, generator=gen, device="cuda") for _ in range(3)]
    sim.init_equilibrium(1.0 + 0.01 * r[0], 0.05 + 0.01 * r[1], 0.02 + 0.01 * r[2])
    return sim


def assert_same_as_single_steps(cls, nx, ny, mode, storage, steps):
    import torch

    ut0 = None
    if mode == "field":
        gen = torch.Generator(device="cuda").manual_seed(7)
        ut0 = torch.randn(2, ny, nx, generator=gen, device="cuda")
    one, many = (_sim(cls, nx, ny, mode, storage, ut0) for _ in range(2))
    for n in steps:
        for _ in range(n):
            one.step(1)
        many.step(n)
        assert one.time == many.time
        assert torch.equal(one.state().view(torch.uint8), many.state().view(torch.uint8)), n
        assert (one.state_ptr() == one._bufs[0].data_ptr()) == (
            many.state_ptr() == many._bufs[0].data_ptr())


# rows of one pack; of 31, 32 and 33 packs (one periodic strip up to 32); a row of exactly 15 strips of 30 packs, of one pack more and one fewer;
# fewer rows than segments; a 16-bit row that 8-node packs do not divide (2052, 1804); 4.2 M
# nodes put both states of every storage type beyond L2
SIZES = [(4, 900001), (128, 25000), (132, 25000), (124, 25001), (1800, 2003), (1804, 2001), (1796, 2003), (131072, 28), (2052, 1801)]


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("mode", ["zero", "fluid", "prescribed", "field"])
@pytest.mark.parametrize("lattice", ["D2Q9", "D2Q9Cascaded"])
def test_several_steps_per_pass_equal_single_steps(lattice, mode, storage):
    import paper_1312_3297_gb300 as pkg

    for nx, ny in SIZES:
        assert_same_as_single_steps(getattr(pkg, lattice), nx, ny, mode, storage, (3, 7))
