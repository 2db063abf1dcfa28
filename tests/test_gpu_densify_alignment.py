"""gs_densify_plan on a P that is only 4-byte aligned: the plan reads single
floats there and decides as on the aligned copy, every flag and count (the
workspace) the same bytes."""
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


@pytest.mark.parametrize("words", [1, 2, 3])
@pytest.mark.parametrize("n", [1, 257, 1000])
def test_plan_off_alignment(n, words):
    g = torch.Generator(device=DEV).manual_seed(n)
    r = lambda *s: torch.rand(s, generator=g, device=DEV)  # noqa: E731
    P = torch.zeros((n, 64), device=DEV)
    P[:, :59] = torch.from_numpy(synth.gaussians_uniform(n, n)).to(DEV)
    P[:, 59] = 12 * r(n) - 8  # volume-mask logits on both sides of logit(0.01)
    cnt = torch.randint(0, 4, (n,), generator=g, device=DEV, dtype=torch.int32)
    stats = lib.grad_stats(acc := r(n) * cnt, rgb := r(n) * cnt, cnt)
    prm = lib.GsDensifyParams(0.5, 9.0, 0, -3.5, -1.0, 1, 2**31 - 1, -2.9, 0.47, 1, -4.595)
    off = torch.zeros(64 * n + words, device=DEV)[words:].view(n, 64)
    off.copy_(P)
    assert P.data_ptr() % 16 == 0 and off.data_ptr() % 16 == 4 * words
    got = []
    for p in (P, off):
        ws = torch.zeros(lib.gs_densify_workspace_bytes(n), dtype=torch.uint8, device=DEV)
        counts = torch.full((4,), -1, dtype=torch.int64, device=DEV)
        lib.gs_densify_plan(n, p, stats, prm, ws, counts)
        got.append((ws, counts))
    torch.cuda.synchronize()
    assert torch.equal(got[0][1], got[1][1]) and torch.equal(got[0][0], got[1][0])
    assert bool((got[0][1] >= 0).all())
    assert acc.numel() == rgb.numel() == n  # held while the struct's pointers are used
    assert lib.gs_get_device_error() == 0
