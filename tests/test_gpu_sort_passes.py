"""The depth order at the sizes where its passes change: counts around a
chunk of 2048 keys and beyond 152 chunks, depths that span few bits (three
passes), many (four) or none, grids of one super-tile, of one pass and of two,
and of so many tiles that their starts take a launch of sums.

Checked without a second sort: every tile's list ascends strictly in (depth,
index), and the (tile, Gaussian) pairs are those of the same call over slices
of the Gaussians, the smallest of which go through a single block (compared with the oracle
in the parity tests). All integers: equality is exact."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, synth  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


def _records(n, W, H, depth, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    r = lambda *s: torch.rand(s, generator=g, device=DEV)  # noqa: E731
    s = torch.zeros((n, 12), device=DEV)
    s[:, 0], s[:, 1] = r(n) * (W + 16) - 8, r(n) * (H + 16) - 8
    s[:, 2] = s[:, 4] = 0.25  # two pixels of standard deviation
    s[:, 5] = 0.9
    s[:, 9] = {"near": 2.0 + 6.0 * r(n), "wide": torch.exp(60 * r(n) - 6), "equal": torch.full((n,), 3.0, device=DEV),
               "few": 1.0 + torch.floor(4 * r(n))}[depth]
    ints = s.view(torch.int32)
    ints[:, 10] = 6
    ints[:, 11] = (r(n) < 0.7).int()  # visible or culled
    ints[ints[:, 11] == 0, 10] = 0
    return s


def _sort(s, cam, capacity):
    n = s.shape[0]
    ws = torch.full((lib.gs_sort_workspace_bytes(n, capacity, cam),), 0xA5, dtype=torch.uint8, device=DEV)
    vals = torch.zeros(max(capacity, 1), dtype=torch.int32, device=DEV)
    ranges = torch.zeros((cam.tiles, 2), dtype=torch.int32, device=DEV)
    count = torch.zeros(1, dtype=torch.int64, device=DEV)
    lib.gs_sort(s, n, cam, ws, capacity, vals, ranges, count)
    P = int(count.item())
    assert P <= capacity and lib.gs_get_device_error() == 0
    r = ranges.long()
    ln = r[:, 1] - r[:, 0]
    assert int(ln.sum()) == P
    tile = torch.repeat_interleave(torch.arange(cam.tiles, device=DEV), ln)
    at = torch.repeat_interleave(r[:, 0] - (torch.cumsum(ln, 0) - ln), ln) + torch.arange(P, device=DEV)
    return tile, vals[at].long()


@pytest.mark.parametrize("n,W,H,tile,depth", [
    (1, 64, 48, 8, "near"), (2925, 600, 400, 8, "near"), (2926, 600, 400, 8, "wide"), (2927, 600, 400, 16, "equal"),
    (70_001, 600, 400, 8, "wide"), (70_001, 600, 400, 8, "few"), (700_003, 900, 700, 16, "near"),
    (20_000, 4000, 3000, 8, "near"), (20_000, 4000, 3000, 8, "wide"), (5_000, 32, 30, 32, "near"),
    (5_000, 250, 200, 32, "equal")])
def test_lists(n, W, H, tile, depth):
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile)
    s = _records(n, W, H, depth, n + W)
    cap = 40 * n + 64
    t, g = _sort(s, cam, cap)
    d = s[:, 9].contiguous().view(torch.int32).long()[g]
    same = t[1:] == t[:-1]
    assert bool(((d[1:] > d[:-1]) | ((d[1:] == d[:-1]) & (g[1:] > g[:-1])) | ~same).all())
    pairs = []
    step = max(1500, n // 40 + 1)
    for a in range(0, n, step):  # slices, the largest sets in 40 of them
        ts, gs = _sort(s[a:a + step].contiguous(), cam, 40 * step + 64)
        pairs.append(ts * n + gs + a)
    assert torch.equal((t * n + g).sort().values, torch.cat(pairs).sort().values)
