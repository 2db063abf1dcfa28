"""Row movement of the densification and the predictor's features at the edges
of warps and blocks.

Densification: survivors, clones and children against their definition
(copies are exact; a child's mean is compared at 1e-5 of the offset's scale, a
few float32 roundings of values of order 1). Features: X and state off 16-byte
alignment must give the bits of the aligned call."""
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


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 1000])
def test_densify_rows(n):
    g = torch.Generator().manual_seed(n)
    r = lambda *s: torch.rand(s, generator=g)  # noqa: E731
    P = torch.zeros((n, 64))
    P[:, :59] = torch.from_numpy(synth.gaussians_uniform(n, n)).float()
    m, v = r(n, 64), r(n, 64)
    frozen = (r(n) < 0.5).to(torch.uint8)
    cnt = torch.randint(0, 4, (n,), generator=g, dtype=torch.int32)
    acc, rgb = r(n) * cnt, r(n) * cnt
    ids = torch.arange(n, dtype=torch.int32)
    low = -1.0
    prm = lib.GsDensifyParams(0.5, 9.0, 0, -3.5, low, 0, 2**31 - 1, 9.0, 0.47)
    z = torch.randn((n, 2, 3), generator=g)
    d = lambda t: t.to(DEV).contiguous()  # noqa: E731
    dev = [d(t) for t in (P, m, v, frozen, acc, rgb, cnt, ids, z)]
    cap = 3 * n + 2
    ws = torch.zeros(lib.gs_densify_workspace_bytes(n), dtype=torch.uint8, device=DEV)
    counts = torch.zeros(4, dtype=torch.int64, device=DEV)
    lib.gs_densify_plan(n, dev[0], lib.grad_stats(dev[4], dev[5], dev[6]), prm, ws, counts)
    o = [torch.full((cap, 64), -7.0, device=DEV) for _ in range(3)]
    fr, carried = torch.full((cap,), 9, dtype=torch.uint8, device=DEV), torch.full((cap,), -1, dtype=torch.int32, device=DEV)
    lib.gs_densify_apply(n, dev[0], dev[1], dev[2], dev[3], [lib.densify_carry(dev[7], carried)], prm, dev[8], ws, cap, *o, fr)
    cand = (cnt > 0) & (acc / cnt.clamp(min=1).float() >= 0.5)
    clone = cand & (P[:, 3:6].amax(1) <= -3.5)
    split, ok = cand & ~clone, ~(P[:, 10] < low)
    keep, kid = ~split & ok, split & ok
    k, c, h = int(keep.sum()), int((clone & ok).sum()), int(kid.sum())
    assert counts.tolist() == [k, c, 2 * h, int(split.sum())]
    P2, m2, v2 = (t.cpu() for t in o)
    assert torch.equal(P2[:k], P[keep]) and torch.equal(m2[:k], m[keep]) and torch.equal(v2[:k], v[keep])
    assert torch.equal(fr.cpu()[:k], frozen[keep]) and torch.equal(carried.cpu()[:k], ids[keep])
    assert torch.equal(P2[k:k + c], P[clone & ok])
    end = k + c + 2 * h
    assert not m2[k:end].any() and not v2[k:end].any() and not fr.cpu()[k:end].any() and not carried.cpu()[k:end].any()
    assert bool((P2[end:] == -7.0).all() and (m2[end:] == -7.0).all() and (fr.cpu()[end:] == 9).all())
    src = P[kid].repeat_interleave(2, 0)
    got = P2[k + c:end]
    assert torch.equal(got[:, 6:], src[:, 6:]) and torch.equal(got[:, 3:6], src[:, 3:6] - torch.tensor(0.47))
    rank = (torch.cumsum(split.long(), 0) - 1)[kid]
    q = src[:, 6:10].double()
    q = q / q.norm(dim=1, keepdim=True)
    s = src[:, 3:6].double().exp() * z[rank].reshape(-1, 3).double()
    t = 2 * torch.linalg.cross(q[:, 1:], s) if h else s
    mean = src[:, :3].double() + s + q[:, :1] * t + (torch.linalg.cross(q[:, 1:], t) if h else s)
    if h:
        assert (got[:, :3].double() - mean).abs().max() <= 1e-5


@pytest.mark.parametrize("n", [1, 33, 257])
def test_features_off_alignment(n):
    g = torch.Generator(device=DEV).manual_seed(n)
    r = lambda *s: torch.rand(s, generator=g, device=DEV)  # noqa: E731
    P, acc, rgb = r(n, 64), r(n), r(n)
    cnt = torch.randint(0, 3, (n,), generator=g, device=DEV, dtype=torch.int32)
    state = r(n, 12)
    X = torch.zeros((n, 16), dtype=torch.bfloat16, device=DEV)
    lib.gs_pred_features(n, P, acc, rgb, cnt, state, 3, 10, 0.2, 0.3, X)
    off = torch.zeros(12 * n + 1, device=DEV)[1:].view(n, 12)  # 4 bytes off
    off.copy_(state)
    X2 = torch.zeros(16 * n + 2, dtype=torch.bfloat16, device=DEV)[2:].view(n, 16)
    for s_, x_ in ((off, torch.zeros_like(X)), (state, X2), (off, X2)):
        x_.zero_()
        lib.gs_pred_features(n, P, acc, rgb, cnt, s_, 3, 10, 0.2, 0.3, x_)
        assert torch.equal(x_.view(torch.int16), X.view(torch.int16))
    assert lib.gs_get_device_error() == 0
