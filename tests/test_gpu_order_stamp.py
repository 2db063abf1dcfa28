"""The tile order that a sort leaves in its workspace is good for that sort's
lists alone: a later sort in the same workspace that makes no order (fewer
than 456 tiles, no Gaussians, no capacity) leaves none behind, and the
rasteriser then takes the tiles ascending. Checked against the calls that take
no workspace, bit for bit in the forward, and in the backward up to the order
of the atomic additions (1e-5 of the largest value)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib, synth  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"
N, W, H = 6000, 640, 400


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


class _Lists:
    def __init__(self, P, cam, cap):
        self.cam, self.cap = cam, cap
        self.splats = torch.zeros((P.shape[0], lib.SPLAT), device=DEV)
        lib.gs_project(P, P.shape[0], 3, cam, self.splats)
        self.vals = torch.zeros(max(cap, 1), dtype=torch.int32, device=DEV)
        self.ranges = torch.zeros((cam.tiles, 2), dtype=torch.int32, device=DEV)
        self.count = torch.zeros(1, dtype=torch.int64, device=DEV)

    def sort(self, ws, n=None):
        lib.gs_sort(self.splats, self.splats.shape[0] if n is None else n, self.cam, ws, self.cap, self.vals,
                    self.ranges, self.count)

    def render(self, ws=None):
        """Image, T, last contributors, gradient; tiles in the workspace's order, or ascending."""
        c = self.cam
        o = [torch.full((3, c.height, c.width), 9.0, device=DEV), torch.full((c.height, c.width), 9.0, device=DEV),
             torch.full((c.height, c.width), -1, dtype=torch.int32, device=DEV)]
        g2 = torch.zeros_like(self.splats)
        dl = torch.ones_like(o[0])
        if ws is None:
            lib.gs_render_fwd_cfg(self.splats, self.vals, self.ranges, c, None, *o)
            lib.gs_raster_bwd_cfg(self.splats, self.vals, self.ranges, c, None, o[1], o[2], dl, None, g2)
        else:
            lib.gs_render_fwd_sorted(self.splats, self.vals, self.ranges, c, None, None, *o, None, None, ws)
            lib.gs_raster_bwd_sorted(self.splats, self.vals, self.ranges, c, None, o[1], o[2], dl, None, None, None, g2,
                                     ws)
        torch.cuda.synchronize()
        return o, g2


@pytest.mark.parametrize("then", ["small grid", "no Gaussians", "no capacity"])
def test_a_later_sort_leaves_no_old_order(then):
    scene = synth.surface_scene(N, N, 2, W, H, seed=3)
    P = torch.zeros((N, 64), device=DEV)
    P[:, :59] = torch.from_numpy(scene.init).to(DEV)
    large = lib.camera(scene.cameras[0], tile=8)
    small = lib.camera(synth.hemisphere_cameras(2, 4.0, 200, 120)[0], tile=8)
    assert large.tiles >= 456 > small.tiles
    a = _Lists(P, large, 200_000)
    later = _Lists(P, small if then == "small grid" else large, 0 if then == "no capacity" else 200_000)
    size = max(lib.gs_sort_workspace_bytes(N, x.cap, x.cam) for x in (a, later))
    ws = torch.zeros(size, dtype=torch.uint8, device=DEV)
    a.sort(ws)
    want, grad = a.render()
    for got in (a.render(ws), None):
        if got is None:
            if then != "small grid":  # what other use of the memory would leave of the order: one tile many times
                ws[256:256 + 4 * large.tiles] = 0
            later.sort(ws, 0 if then == "no Gaussians" else None)
            got = a.render(ws)
        for x, y in zip(got[0], want):
            assert torch.equal(x, y)
        assert (got[1] - grad).abs().max() <= 1e-5 * grad.abs().max()
    lib.gs_get_device_error()  # no capacity raises its flag
