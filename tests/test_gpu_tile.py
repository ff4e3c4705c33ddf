"""Several steps per launch on shared-memory tiles (automatic kernel variant, lattices whose
states stay in L2, and rows that no vector pack divides) against the same steps taken one call
at a time: the same states bit for bit, in the same buffer."""
import pytest
from test_gpu_march import assert_same_as_single_steps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# lattices smaller than a tile's halo (wrapped several times), one tile, ragged last tiles, odd
# heights, long and flat ones, pack widths 1, 2, 4 and 8; the last one's states exceed L2
SIZES = [(1, 1), (1, 9), (9, 1), (2, 3), (63, 41), (64, 64), (33, 130), (130, 77), (300, 36),
         (36, 300), (1001, 20), (257, 511), (520, 260), (1451, 2899)]


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("mode", ["zero", "fluid", "prescribed", "field"])
@pytest.mark.parametrize("lattice", ["D2Q9", "D2Q9Cascaded"])
def test_tiles_equal_single_steps(lattice, mode, storage):
    import paper_1312_3297_gb300 as pkg

    for nx, ny in SIZES:
        steps = (5, 6, 7, 12, 25) if nx * ny < 100000 else (7, 8)
        assert_same_as_single_steps(getattr(pkg, lattice), nx, ny, mode, storage, steps)
