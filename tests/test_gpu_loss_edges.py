"""The Eq. 3 loss and its gradient at the edges of its 32 x 32 tiles against
float64 PyTorch.

Tolerances (set before the first run): a window sum of 121 float32 products of
values up to 1 is off by about 1e-6 of its size at most; the map divides by at
least C2 = 9e-4 and the gradient's terms are of the size of its largest value,
so 1e-6 / 9e-4, about 1e-3 of the largest gradient, bounds it; the mean over the
image of the map and of |x - y| is compared at 1e-5."""
import math

import pytest

torch = pytest.importorskip("torch")

from paper_2504_06716_gb300 import lib  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06716_gb300 import build

    build.build()
    lib.load()


def _reference(x, y, lam):
    x = x.double().requires_grad_(True)
    y = y.double()
    w = torch.tensor([math.exp(-(k - 5) ** 2 / 4.5) for k in range(11)], dtype=torch.float64)
    w = w / w.sum()

    def win(t):
        t = torch.nn.functional.conv2d(t[:, None], w.view(1, 1, 1, 11), padding=(0, 5))
        return torch.nn.functional.conv2d(t, w.view(1, 1, 11, 1), padding=(5, 0))[:, 0]

    mx, my = win(x), win(y)
    vx, vy, c = win(x * x) - mx * mx, win(y * y) - my * my, win(x * y) - mx * my
    ssim = ((2 * mx * my + 1e-4) * (2 * c + 9e-4)) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
    loss = (1 - lam) * (x - y).abs().mean() + lam * (1 - ssim.mean())
    (g,) = torch.autograd.grad(loss, x)
    return loss.item(), g


@pytest.mark.parametrize("H,W", [(1, 1), (3, 40), (31, 33), (32, 32), (33, 64), (64, 31), (37, 129), (500, 333)])
@pytest.mark.parametrize("lam", [0.0, 0.2, 1.0])
def test_edges(H, W, lam):
    g = torch.Generator().manual_seed(H * 1000 + W)
    y = torch.rand((3, H, W), generator=g)
    x = (y + 0.1 * torch.randn((3, H, W), generator=g)).clamp(0, 1)
    ref, gref = _reference(x, y, lam)
    ws = torch.full((lib.gs_loss_workspace_bytes(H, W),), 0xA5, dtype=torch.uint8, device=DEV)
    loss, dl = torch.zeros(1, device=DEV), torch.full((3, H, W), 7.0, device=DEV)
    for _ in range(2):  # the workspace as it comes, and as the call leaves it
        lib.gs_loss(x.to(DEV), y.to(DEV), H, W, lam, ws, loss, dl)
        assert abs(loss.item() - ref) <= 1e-5
        ok = x != y
        assert (dl.cpu().double() - gref)[ok].abs().max() <= 1e-3 * gref.abs().max()
    assert lib.gs_get_device_error() == 0
