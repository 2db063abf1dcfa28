"""The resume record where a tile's rays all stop inside its list, in front of
unfrozen entries that no ray reaches: the resuming backward against the plain
one and a float64 compositor.

Nothing that was blended may lose its gradient: resume_pos lies behind every
unfrozen entry in front of the tile's deepest last contributor, and the
gradients are the plain backward's. Lists of 512 entries whose rays stop after
about 8, 50 or 150 of them, in tiles of one and of several 8-pixel blocks,
with blocks that stop far apart, for every batch size and freeze map.

Tolerances (set before the first run): the image is the plain forward's bit
for bit, as are record and position across pixels per thread and batch size;
gradients within 1e-3 of their block's largest value, as elsewhere in this
suite (T recovered backward through up to 512 divisions by 1 - alpha <= 0.99,
each off by at most 100 * 2^-24 relative where alpha is 0.99 and by 2^-23
where it is below 0.5: 512 * 2^-23 = 6.1e-5, or 8 * 100 * 2^-24 = 4.8e-5)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, synth  # noqa: E402

import test_gpu_raster_blocks as rb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"
N = 512
BATCHES = (32, 64, 128, 256)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


def _scene(tile, depth, apart, seed):
    """Splats wider than the tile, of the opacity that stops a ray after about `depth` of
    them; apart: every second one reaches the left 8 columns alone, which stop first."""
    g = torch.Generator().manual_seed(seed)
    r = lambda *s: torch.rand(s, generator=g)  # noqa: E731
    spl = rb._splats(N, tile, seed, False)
    spl[:, 2:5] /= tile  # radii of sqrt(tile) to 8 sqrt(tile) px
    lo = {8: 0.6, 50: 0.14, 150: 0.065}[depth]
    spl[:, 5] = lo * (1.0 + 0.5 * r(N))
    if apart:
        spl[::2, 0] = 3.0 * r(N // 2)
        spl[::2, 2], spl[::2, 3], spl[::2, 4] = 1.0, 0.0, 0.01  # 1 px by 10: nothing past column 8
    return spl


def _freeze(kind):
    if kind is None:
        return None
    g = torch.Generator().manual_seed(7)
    return (torch.rand(N, generator=g) < kind).to(torch.uint8)


@pytest.mark.parametrize("frozen_frac", [None, 0.4, 0.9])
@pytest.mark.parametrize("depth", [8, 50, 150])
@pytest.mark.parametrize("tile,apart", [(8, False), (16, False), (16, True), (32, True)])
def test_rays_that_stop_in_front_of_unfrozen_entries(tile, apart, depth, frozen_frac):
    W, H, bg = tile, tile, (0.1, 0.4, 0.2)
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile, bg=bg)
    spl = _scene(tile, depth, apart, 10 * tile + depth)
    frozen = _freeze(frozen_frac)
    dl = torch.randn((3, H, W), generator=torch.Generator().manual_seed(depth))
    d = lambda t: None if t is None else t.to(DEV).contiguous()  # noqa: E731
    dspl, ddl, dfr = d(spl), d(dl), d(frozen)
    vals = torch.arange(N, dtype=torch.int32, device=DEV)
    ranges = torch.tensor([[0, N]], dtype=torch.int32, device=DEV)

    def out():
        return [torch.full((3, H, W), 9.0, device=DEV), torch.full((H, W), 9.0, device=DEV),
                torch.full((H, W), -1, dtype=torch.int32, device=DEV)]

    plain, g_plain = out(), torch.zeros((N, 12), device=DEV)
    lib.gs_render_fwd_cfg(dspl, vals, ranges, cam, None, *plain)
    lib.gs_raster_bwd_cfg(dspl, vals, ranges, cam, None, plain[1], plain[2], ddl, dfr, g_plain)
    deep = int(plain[2].max())
    assert 0 < deep < N - 32, "some ray runs through the whole list"
    awake = torch.ones(N, dtype=torch.bool) if frozen is None else frozen == 0
    assert bool(awake[deep + 1:].any()), "no unfrozen entry behind the stop"
    passed = torch.nonzero(awake[:deep]).flatten()
    first = None
    for ppt in (1, 2, 4) if tile >= 16 else (1, 2):
        for batch in BATCHES:
            cfg, o = lib.raster_config(ppt, batch), out()
            rs = torch.full((H * W * 4,), float("nan"), device=DEV)
            rp = torch.full((1,), -1, dtype=torch.int32, device=DEV)
            lib.gs_render_fwd_resume(dspl, vals, ranges, cam, cfg, dfr, *o, rs, rp)
            g2 = torch.zeros((N, 12), device=DEV)
            lib.gs_raster_bwd_resume(dspl, vals, ranges, cam, cfg, o[1], o[2], ddl, dfr, rs, rp, g2)
            for a, b in zip(o, plain):
                assert torch.equal(a, b), (ppt, batch)
            p = int(rp)
            if passed.numel():
                assert p > int(passed[-1]) and awake[p - 1], (ppt, batch, p)
            for cols in (slice(0, 2), slice(2, 5), slice(5, 6), slice(6, 9)):
                want = g_plain[:, cols]
                assert (g2[:, cols] - want).abs().max() <= 1e-3 * want.abs().max(), (ppt, batch, cols)
            if first is None:
                first = (rs.clone(), p, g2.cpu().double())
            assert torch.equal(rs, first[0]) and p == first[1], (ppt, batch)
    near, grad = rb._reference(spl, N, W, H, bg, dl, torch.zeros(N) if frozen is None else frozen)[3:]
    if not near.any():  # a decision taken the other way changes everything in front of it
        for cols in (slice(0, 2), slice(2, 5), slice(5, 6), slice(6, 9)):
            assert (first[2][:, cols] - grad[:, cols]).abs().max() <= 1e-3 * grad[:, cols].abs().max(), cols
    assert lib.gs_get_device_error() == 0
