"""Splats too faint to be blended anywhere in a caller's own lists (opacity 0,
subnormal, negative or below 1/255) in the rasteriser backward: they get no
gradient, and their neighbours in the list get what they get with those
splats moved out of sight (to 1e-5 of the largest value: the pairs in which
splats are summed are the same, only other lanes' zeros are added)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, synth  # noqa: E402

import test_gpu_raster_blocks as rb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


@pytest.mark.parametrize("frozen_frac", [0.0, 0.5])
@pytest.mark.parametrize("tile,ppt", [(8, 1), (8, 2), (16, 1), (16, 4), (32, 2)])
@pytest.mark.parametrize("opacity", [0.0, -0.0, 1e-40, -0.5, 0.0039])
def test_a_faint_splat_gets_nothing(tile, ppt, opacity, frozen_frac):
    n, W, H = 37, tile, tile
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile)
    spl = rb._splats(n, tile, tile + ppt, False)
    faint = [0, 5, 20, 36]
    g = torch.Generator().manual_seed(ppt)
    dl = torch.randn((3, H, W), generator=g)
    frozen = (torch.rand(n, generator=g) < frozen_frac).to(torch.uint8)
    frozen[faint] = 0
    d = lambda t: t.to(DEV).contiguous()  # noqa: E731
    vals = torch.arange(n, dtype=torch.int32, device=DEV)
    ranges = torch.tensor([[0, n]], dtype=torch.int32, device=DEV)
    cfg = lib.raster_config(ppt, 64)
    got = []
    for seen in (True, False):
        s = spl.clone()
        if seen:
            s[faint, 5] = opacity
        else:
            s[faint, 0:2] = 1e6
            s[faint, 2:5] = torch.tensor([1.0, 0.0, 1.0])
        img, tf = torch.zeros((3, H, W), device=DEV), torch.zeros((H, W), device=DEV)
        nl = torch.zeros((H, W), dtype=torch.int32, device=DEV)
        lib.gs_render_fwd_cfg(d(s), vals, ranges, cam, cfg, img, tf, nl)
        g2 = torch.zeros((n, 12), device=DEV)
        lib.gs_raster_bwd_cfg(d(s), vals, ranges, cam, cfg, tf, nl, d(dl), d(frozen), g2)
        got.append((img.cpu(), tf.cpu(), g2.cpu()))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert not got[0][2][faint].any() and bool(torch.isfinite(got[0][2]).all())
    for cols in (slice(0, 2), slice(2, 5), slice(5, 6), slice(6, 9)):
        want = got[1][2][:, cols]
        assert (got[0][2][:, cols] - want).abs().max() <= 1e-5 * want.abs().max(), cols
    assert lib.gs_get_device_error() == 0
