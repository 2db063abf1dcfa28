"""Records with a value that is not finite in the rasteriser backward: a mean
or conic that is not finite is never blended, so its splat gets no gradient
and its neighbours in the list get what they get without it (to 1e-5 of the
largest value: the scalar steps against the packed ones)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, synth  # noqa: E402

import test_gpu_raster_blocks as rb  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"
NAN, INF = float("nan"), float("inf")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


@pytest.mark.parametrize("tile,ppt", [(8, 1), (8, 2), (16, 1), (16, 4), (32, 2)])
@pytest.mark.parametrize("column,value", [(0, NAN), (0, INF), (1, -INF), (2, NAN), (3, NAN), (3, INF), (4, INF)])
def test_a_splat_without_a_finite_shape_gets_nothing(tile, ppt, column, value):
    n, W, H = 37, tile, tile
    cam = lib.camera(synth.pinhole(W, H, 60.0, (0, 0, -4.0), up=(0, 1, 0)), tile=tile)
    spl = rb._splats(n, tile, tile + ppt, False)
    bad = [0, 5, 20, 36]  # next to blended ones, on both sides of the first 32
    dl = torch.randn((3, H, W), generator=torch.Generator().manual_seed(ppt))
    d = lambda t: t.to(DEV).contiguous()  # noqa: E731
    vals = torch.arange(n, dtype=torch.int32, device=DEV)
    ranges = torch.tensor([[0, n]], dtype=torch.int32, device=DEV)
    cfg = lib.raster_config(ppt, 64)
    got = []
    for odd in (False, True):
        s = spl.clone()
        if odd:
            s[bad, column] = value
        else:
            s[bad, 5] = 0.0  # the same list without them: no alpha reaches 1/255
        img, tf = torch.zeros((3, H, W), device=DEV), torch.zeros((H, W), device=DEV)
        nl = torch.zeros((H, W), dtype=torch.int32, device=DEV)
        lib.gs_render_fwd_cfg(d(s), vals, ranges, cam, cfg, img, tf, nl)
        g2 = torch.zeros((n, 12), device=DEV)
        lib.gs_raster_bwd_cfg(d(s), vals, ranges, cam, cfg, tf, nl, d(dl), None, g2)
        got.append((img.cpu(), tf.cpu(), nl.cpu(), g2.cpu()))
    for a, b in zip(got[0][:3], got[1][:3]):
        assert torch.equal(a, b)
    assert not got[1][3][bad].any() and bool(torch.isfinite(got[1][3]).all())
    for cols in (slice(0, 2), slice(2, 5), slice(5, 6), slice(6, 9)):
        want = got[0][3][:, cols]
        assert (got[1][3][:, cols] - want).abs().max() <= 1e-5 * want.abs().max(), cols
    assert lib.gs_get_device_error() == 0
