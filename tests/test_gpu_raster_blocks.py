"""The rasteriser's warps on one tile against a float64 PyTorch compositor:
list lengths around the 32 entries a warp stages and the splats it blends
together, splats that miss some of a tile's blocks, rays that stop inside a
group, needle-thin conics, every tile size and pixels-per-thread.

Tolerances (set before the first run): at most 70 terms are summed per pixel
in float32, each with a relative error below 8 * 2^-24 (exponent, exp, two
products), so values of order 1 are off by less than 70 * 8 * 2^-24 = 3.4e-5;
1e-4 is asked. Gradients sum such terms over the pixels of a tile and are
compared at 1e-3 of the block's largest value, as elsewhere in this suite.
Pixels with a decision (alpha against 1/255, T against 1e-4) within 1e-5
relative of its threshold are left out of the image comparison, and a case
has few of them."""
import numpy as np
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


def _splats(n, tile, seed, thin):
    """n records around a tile's pixels: means up to 6 px outside it, radii of 1 to 8 px (thin: 0.6 by 40)."""
    g = torch.Generator().manual_seed(seed)
    r = lambda *s: torch.rand(s, generator=g, dtype=torch.float64)  # noqa: E731
    mean = r(n, 2) * (tile + 12) - 6
    s = torch.stack([torch.full((n,), 0.6, dtype=torch.float64), 5 + 35 * r(n)], 1) if thin else 1 + 7 * r(n, 2)
    a = r(n) * np.pi
    R = torch.stack([torch.cos(a), -torch.sin(a), torch.sin(a), torch.cos(a)], 1).view(n, 2, 2)
    Q = R @ torch.diag_embed(1 / s**2) @ R.transpose(1, 2)
    out = torch.zeros((max(n, 1), 12), dtype=torch.float32)
    out[:n, 0:2] = mean.float()
    out[:n, 2], out[:n, 3], out[:n, 4] = Q[:, 0, 0].float(), Q[:, 0, 1].float(), Q[:, 1, 1].float()
    out[:n, 5] = (0.05 + 0.94 * r(n)).float()
    out[:n, 6:9] = r(n, 3).float()
    return out


def _reference(spl, n, W, H, bg, dl, frozen):
    """Image, T, last contributor, near-threshold pixels, gradient [n, 9] in float64."""
    s = spl[:n, :9].double().requires_grad_(True)
    y, x = torch.meshgrid(torch.arange(H), torch.arange(W), indexing="ij")
    T = torch.ones((H, W), dtype=torch.float64)
    C = torch.zeros((3, H, W), dtype=torch.float64)
    last = torch.zeros((H, W), dtype=torch.int64)
    done = torch.zeros((H, W), dtype=torch.bool)
    near = torch.zeros((H, W), dtype=torch.bool)
    for j in range(n):
        dx, dy = s[j, 0] - x, s[j, 1] - y
        power = -0.5 * (s[j, 2] * dx * dx + s[j, 4] * dy * dy) - s[j, 3] * dx * dy
        oG = s[j, 5] * torch.exp(power)
        al = torch.clamp(oG, max=0.99)
        use = ~done & (power <= 0) & (al >= 1 / 255)
        tn = T * (1 - al)
        near |= ~done & ((al * 255 - 1).abs() < 1e-5)
        near |= use & ((tn * 1e4 - 1).abs() < 1e-5)
        done = done | (use & (tn < 1e-4))
        add = use & ~(tn < 1e-4)
        w = torch.where(add, al * T, torch.zeros_like(T))
        C = C + w * s[j, 6:9, None, None]
        T = torch.where(add, tn, T)
        last = torch.where(add, torch.full_like(last, j + 1), last)
    img = C + T * torch.tensor(bg, dtype=torch.float64)[:, None, None]
    grad = torch.zeros((n, 9), dtype=torch.float64)
    if n and img.requires_grad:
        (grad,) = torch.autograd.grad((img * dl.double()).sum(), s)
        grad[frozen[:n] != 0] = 0
    return img.detach(), T.detach(), last, near, grad


CASES = [(t, p, n, thin) for t, ps in ((8, (1, 2)), (16, (1, 2, 4)), (32, (1, 2, 4))) for p in ps
         for n, thin in ((0, False), (1, False), (3, False), (5, False), (31, True), (32, False), (33, False), (70, False),
                         (70, True))]


@pytest.mark.parametrize("tile,ppt,n,thin", CASES)
def test_one_tile_against_float64(tile, ppt, n, thin):
    W, H, bg = tile - 1, tile - 2, (0.1, 0.4, 0.2)  # ragged: some lanes are outside the image
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile, bg=bg)
    spl = _splats(n, tile, 100 * tile + 10 * n + thin, thin)
    g = torch.Generator().manual_seed(n)
    dl = torch.randn((3, H, W), generator=g)
    frozen = (torch.rand(max(n, 1), generator=g) < 0.4).to(torch.uint8)
    img, T, last, near, grad = _reference(spl, n, W, H, bg, dl, frozen)
    assert near.float().mean() < 0.02
    d = lambda t: t.to(DEV).contiguous()  # noqa: E731
    vals = torch.arange(max(n, 1), dtype=torch.int32, device=DEV)
    ranges = torch.tensor([[0, n]], dtype=torch.int32, device=DEV)
    o = [torch.full((3, H, W), 9.0, device=DEV), torch.full((H, W), 9.0, device=DEV),
         torch.full((H, W), -1, dtype=torch.int32, device=DEV)]
    cfg = lib.raster_config(ppt, 64)
    lib.gs_render_fwd_cfg(d(spl), vals, ranges, cam, cfg, *o)
    ok = ~near
    assert (o[0].cpu().double() - img).abs()[:, ok].max() <= 1e-4
    assert (o[1].cpu().double() - T).abs()[ok].max() <= 1e-4
    assert torch.equal(o[2].cpu().long()[ok], last[ok])
    if near.any():  # a decision taken the other way changes the gradient of everything in front of it
        return
    g2 = torch.zeros((max(n, 1), 12), device=DEV)
    lib.gs_raster_bwd_cfg(d(spl), vals, ranges, cam, cfg, o[1], o[2], d(dl), d(frozen), g2)
    got = g2.cpu().double()[:n]
    for cols in (slice(0, 2), slice(2, 5), slice(5, 6), slice(6, 9)):
        if n:
            assert (got[:, cols] - grad[:, cols]).abs().max() <= 1e-3 * max(float(grad[:, cols].abs().max()), 1e-6), cols
    assert not g2[:, 9:].any() and not got[frozen[:n] != 0].any()
    assert lib.gs_get_device_error() == 0


@pytest.mark.parametrize("tile,ppt", [(8, 1), (8, 2), (16, 2), (16, 4), (32, 1)])
def test_a_pixel_without_a_finite_gradient_stays_by_itself(tile, ppt):
    """NaN in dL/dC of one pixel reaches the splats blended there and no others
    (those: equal to the gradient without that pixel, up to float32 rounding
    of the scalar steps against the packed ones, 1e-5 of the largest value)."""
    n, W, H = 70, tile, tile
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile)
    spl = _splats(n, tile, tile + ppt, False)
    dl = torch.randn((3, H, W), generator=torch.Generator().manual_seed(ppt))
    y, x = H // 2, W // 3
    with torch.no_grad():
        dx, dy = spl[:n, 0].double() - x, spl[:n, 1].double() - y
        power = -0.5 * (spl[:n, 2] * dx * dx + spl[:n, 4] * dy * dy) - spl[:n, 3] * dx * dy
        al = torch.clamp(spl[:n, 5] * torch.exp(power), max=0.99)
    d = lambda t: t.to(DEV).contiguous()  # noqa: E731
    vals = torch.arange(n, dtype=torch.int32, device=DEV)
    ranges = torch.tensor([[0, n]], dtype=torch.int32, device=DEV)
    cfg = lib.raster_config(ppt, 64)
    img, tf = torch.zeros((3, H, W), device=DEV), torch.zeros((H, W), device=DEV)
    nl = torch.zeros((H, W), dtype=torch.int32, device=DEV)
    lib.gs_render_fwd_cfg(d(spl), vals, ranges, cam, cfg, img, tf, nl)
    got = []
    for v in (0.0, float("nan")):
        e = dl.clone()
        e[:, y, x] = v
        g2 = torch.zeros((n, 12), device=DEV)
        lib.gs_raster_bwd_cfg(d(spl), vals, ranges, cam, cfg, tf, nl, d(e), None, g2)
        got.append(g2.cpu())
    last = int(nl[y, x].item())
    apart = (al < 0.999 / 255) | (torch.arange(n) >= last)  # certainly not blended at the pixel
    there = (al > 1.001 / 255) & (torch.arange(n) < last) & (power < -1e-6)
    assert apart.any() and there.any()
    assert torch.isnan(got[1][there, 6:9]).all()
    for cols in (slice(0, 2), slice(2, 5), slice(5, 6), slice(6, 9)):
        assert (got[1][apart][:, cols] - got[0][apart][:, cols]).abs().max() <= 1e-5 * got[0][:, cols].abs().max()
