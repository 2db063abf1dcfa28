"""The order in which the rasteriser takes the tiles, at the grid sizes where it
changes: no order below 456 tiles, one block of 1024 tiles or several.

The orders are permutations of the tiles with lengths descending by bucket
(eight to an octave); the forward's results do not depend on the order at all, the
backward's only by the order of its atomic additions; a workspace that another
grid's sort left, an unsorted one and none at all give the same results."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, pipeline, synth  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


def _front(ws, tiles):
    each = (4 * tiles + 255) // 256 * 256
    w = ws[: 256 + 3 * each].cpu().view(torch.int32)
    part = lambda k: w[64 + k * each // 4: 64 + k * each // 4 + tiles].long()  # noqa: E731
    return w[:2].tolist(), part(0), part(1), part(2)


def _bucket(n):
    return torch.where(n > 0, 1 + ((n.float().view(torch.int32) - 0x3F800000) >> 20).long(), 0 * n)


def _descending(order, n, tiles):
    assert torch.equal(order.sort().values, torch.arange(tiles))
    b = _bucket(n)[order]
    assert bool((b[1:] <= b[:-1]).all())


@pytest.mark.parametrize("W,H,tile", [(24 * 16, 18 * 16 + 5, 16), (304, 183, 8), (57 * 8, 8 * 8, 8), (1024, 1024, 32),
                                      (300, 251, 8), (640, 480, 8)])
def test_orders_and_results(W, H, tile):
    scene = synth.surface_scene(6000, 8000, 2, W, H, seed=3)
    cam = lib.camera(scene.cameras[0], tile=tile)
    tiles = cam.tiles
    m = pipeline.Model(scene.init, device=DEV)
    m.frozen[: m.n : 3] = 1
    m.freeze_update(0.0, 0.0, 3)
    v = m.make_view(cam, m.measure_capacity([cam]))
    gt = torch.rand((3, H, W), device=DEV)
    m.rasterize(v)
    stamp, order, _, _ = _front(v.sort_ws, tiles)
    length = (v.ranges[:, 1] - v.ranges[:, 0]).long().cpu()
    if tiles >= 456:
        assert stamp == [cam.width // tile + (cam.width % tile > 0) | -(-cam.height // tile) << 16, 0x67530000 | tile]
        _descending(order, length, tiles)
    else:
        assert stamp == [0, 0]
    m.loss(v, gt)
    img, nl, tf = v.image.clone(), v.n_last.clone(), v.t_final.clone()
    rec, pos = v.resume.clone(), v.resume_pos.clone()
    m.raster_bwd(v)
    grad = m.grad2d.clone()
    m.grad2d.zero_()
    scale = grad.abs().max().item()
    own = v.sort_ws.clone()
    other = own.clone()
    other[:8] = torch.tensor([9, 9, 9, 9, 9, 9, 9, 9], dtype=torch.uint8)  # another grid's
    other[256:2048] = 0xEE
    for ws in (other, torch.full_like(own, 0xA5), own[:512], None):
        for t in (v.image, v.t_final, v.resume):
            t.fill_(-1.0)
        if ws is None:
            lib.gs_render_fwd_resume(m.splats, v.vals, v.ranges, cam, None, m.frozen, v.image, v.t_final, v.n_last,
                                     v.resume, v.resume_pos)
            lib.gs_raster_bwd_resume(m.splats, v.vals, v.ranges, cam, None, v.t_final, v.n_last, v.dl, m.frozen,
                                     v.resume, v.resume_pos, m.grad2d)
        else:
            lib.gs_render_fwd_sorted(m.splats, v.vals, v.ranges, cam, None, m.frozen, v.image, v.t_final, v.n_last,
                                     v.resume, v.resume_pos, ws)
            lib.gs_raster_bwd_sorted(m.splats, v.vals, v.ranges, cam, None, v.t_final, v.n_last, v.dl, m.frozen,
                                     v.resume, v.resume_pos, m.grad2d, ws)
        for a, b in ((v.image, img), (v.n_last, nl), (v.t_final, tf), (v.resume, rec), (v.resume_pos, pos)):
            assert torch.equal(a, b)
        assert (m.grad2d - grad).abs().max().item() <= 1e-5 * scale
        m.grad2d.zero_()
    # a training step: the forward's order and the backward's, by the depth reached
    m.train_step(v, gt, pipeline.default_lrs(4.4))
    torch.cuda.synchronize()
    assert torch.equal(v.image, img) and torch.equal(v.n_last, nl)
    if tiles >= 456:
        _, order, depth, deep = _front(v.sort_ws, tiles)
        ty, tx = -(-H // tile), -(-W // tile)
        pad = torch.zeros((ty * tile, tx * tile), dtype=torch.int32)
        pad[:H, :W] = v.n_last.cpu().view(H, W)
        want = pad.view(ty, tile, tx, tile).amax((1, 3)).flatten().long()
        assert torch.equal(depth, want)
        _descending(order, length, tiles)
        _descending(deep, depth, tiles)
    assert lib.gs_get_device_error() == 0
