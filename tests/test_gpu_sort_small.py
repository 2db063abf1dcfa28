"""The depth order of few Gaussians, sorted by one block, against the same
Gaussians sorted by the passes of many blocks: a set of up to 8192 and the same
set followed by culled ones, which puts it past that size. Counts around a
warp's piece and the block's size, depths that span few bits, many or none. All
integers: equality is exact."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, synth  # noqa: E402
from test_gpu_sort_passes import _records, _sort  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


@pytest.mark.parametrize("n", [1, 31, 33, 1000, 1023, 1025, 1500, 4099, 8191, 8192])
@pytest.mark.parametrize("depth", ["near", "wide", "equal", "few"])
@pytest.mark.parametrize("seen", [1.0, 0.7])
def test_one_block_orders_as_many_do(n, depth, seen):
    W, H, tile = 300, 200, 8
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile)
    s = _records(n, W, H, depth, n)
    if seen == 1.0:
        s.view(torch.int32)[:, 10:] = torch.tensor([6, 1], dtype=torch.int32, device=DEV)
    more = torch.zeros((9000, 12), device=DEV)  # culled
    cap = 40 * n + 64
    small, large = _sort(s, cam, cap), _sort(torch.cat([s, more]), cam, cap)
    assert torch.equal(small[0], large[0]) and torch.equal(small[1], large[1])
