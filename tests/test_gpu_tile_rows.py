"""The tiles that list a splat, decided a row of tiles at a time, against the
tile-by-tile test over the splat's whole rectangle: the same float32 operations
in PyTorch, one rounding each, so the (tile, Gaussian) pairs are equal exactly.

Round, long and needle-like conics (both sides of the bounds up to which a row
is decided at once), opacities down to the listing limit, splats without
dilation, far outside the image and with means that are not finite, and
ellipses that end at a tile's edge up to parts in 10^2 .. 10^7."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, synth  # noqa: E402
from test_gpu_sort_passes import _sort  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


def _records(n, W, H, tile, shape, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    r = lambda *s: torch.rand(s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    big, ratio = {"round": (4.0, 1.5), "long": (30.0, 20.0), "needle": (60.0, 300.0), "tiny": (0.3, 30.0),
                  "any": (200.0, 60.0)}[shape]
    s1 = torch.exp(r(n) * 3.0) / 20.1 * big  # standard deviations along the axes
    s2 = s1 / ratio ** r(n)
    th = r(n) * 6.2831853
    co, si = torch.cos(th), torch.sin(th)
    dil = 0.0 if shape == "tiny" else 0.3
    xx, yy = (s1 * co) ** 2 + (s2 * si) ** 2 + dil, (s1 * si) ** 2 + (s2 * co) ** 2 + dil
    xy = (s1 ** 2 - s2 ** 2) * co * si
    det = xx * yy - xy * xy
    op = torch.where(r(n) < 0.5, r(n), (1.0 + 0.02 * r(n)) / 255.0)
    tau = 2.0 * torch.log(torch.clamp(255.0 * op, min=1.0))
    tau = tau + 1e-3 * (1.0 + tau)
    x, y = r(n) * (W + 80) - 40, r(n) * (H + 80) - 40
    # half of the splats end at a tile's edge, horizontally or vertically, almost
    off = (r(n) - 0.5) * 10.0 ** (-2.0 - 5.0 * r(n))
    edge = torch.floor(r(n) * W / tile) * tile
    x = torch.where(r(n) < 0.25, edge - torch.sqrt(tau * xx) * (1.0 + off), x)
    x = torch.where(r(n) < 0.25, edge - 1.0 + torch.sqrt(tau * xx) * (1.0 + off), x)
    y = torch.where(r(n) < 0.25, edge - torch.sqrt(tau * yy) * (1.0 + off), y)
    s = torch.zeros((n, 12), device=DEV)
    s[:, 0], s[:, 1] = x.float(), y.float()
    s[:, 2], s[:, 3], s[:, 4], s[:, 5] = (yy / det).float(), (-xy / det).float(), (xx / det).float(), op.float()
    if shape == "any":
        s[:: 97, 0] = float("nan")
        s[5:: 97, 1] = 30000.0
        s[7:: 97, 0] = -40000.0
    s[:, 9] = (2.0 + 6.0 * r(n)).float()
    ints = s.view(torch.int32)
    ints[:, 10] = torch.ceil(3.0 * torch.sqrt(torch.maximum(xx, yy))).int() + 1
    ints[:, 11] = 1
    return s


def _ln(x):
    b = x.view(torch.int32)
    e = ((b >> 23) & 0xFF) - 127
    m = ((b & 0x007FFFFF) | 0x3F800000).view(torch.float32)
    s = (m - 1.0) / (m + 1.0)
    s2 = s * s
    p = torch.full_like(s, 0.0666666667)
    for k in (0.0769230769, 0.0909090909, 0.111111111, 0.142857143, 0.2, 0.333333333, 1.0):
        p = p * s2 + k
    return e.float() * 0.693147181 + (2.0 * s) * p


def _expected(s, cam, tile):
    """The pairs of the tile test over each splat's 3-sigma rectangle."""
    n = s.shape[0]
    mx, my, a, b, c, op = (s[:, k].contiguous() for k in range(6))
    rad = s.view(torch.int32)[:, 10].float()
    tx, ty = (cam.width + tile - 1) // tile, (cam.height + tile - 1) // tile
    f = lambda v: torch.floor(v * (1.0 / tile))  # noqa: E731
    big = lambda v, hi: torch.nan_to_num(v, nan=0.0).clamp(-1e6, 1e6).clamp(max=hi)  # noqa: E731
    x0, x1 = big(f(mx - rad), 1e6).clamp(min=0), big(f(mx + rad), tx - 1)
    y0, y1 = big(f(my - rad), 1e6).clamp(min=0), big(f(my + rad), ty - 1)
    w, h = (x1 - x0 + 1).clamp(min=0).long(), (y1 - y0 + 1).clamp(min=0).long()
    x255 = op * 255.0
    tau = 2.0 * _ln(x255)
    tau = tau + 1e-3 * (1.0 + tau)
    cnt = torch.where((x255 >= 1.0) & torch.isfinite(mx) & torch.isfinite(my), w * h, torch.zeros_like(w))
    i = torch.repeat_interleave(torch.arange(n, device=DEV), cnt)
    k = torch.arange(i.numel(), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[i]
    x, y = x0[i].long() + k % w[i], y0[i].long() + k // w[i]
    mx, my, a, b, c, tau = mx[i], my[i], a[i], b[i], c[i], tau[i]
    bx0, by0 = (x * tile).float(), (y * tile).float()
    bx1, by1 = bx0 + (tile - 1), by0 + (tile - 1)

    def quad(dx, dy):
        return ((a * dx) * dx + ((2.0 * b) * dx) * dy) + (c * dy) * dy

    hit = (mx >= bx0) & (mx <= bx1) & (my >= by0) & (my <= by1)
    for ex, ey in ((bx0, by0), (bx1, by1)):
        dx, dy = ex - mx, ey - my
        yo, xo = my - (b / c) * dx, mx - (b / a) * dy
        hit |= quad(dx, torch.minimum(torch.maximum(yo, by0), by1) - my) <= tau
        hit |= quad(torch.minimum(torch.maximum(xo, bx0), bx1) - mx, dy) <= tau
    return ((y * tx + x) * n + i)[hit].sort().values


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("shape", ["round", "long", "needle", "tiny", "any"])
def test_rows_decide_as_tiles_do(tile, shape):
    n, W, H = 30_000, 1237, 822
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile)
    s = _records(n, W, H, tile, shape, tile + len(shape))
    want = _expected(s, cam, tile)
    assert want.numel() > n // 8
    t, g = _sort(s, cam, 2 * want.numel() + 4 * n + 64)
    got = (t * n + g).sort().values
    assert torch.equal(got, want)
