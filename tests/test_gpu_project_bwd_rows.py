"""The projection backward over lists of any length: a warp takes 32 entries
and moves their rows through shared memory, so a list's remainder, culled
entries among seen ones, both write modes and both statistics windows are
checked entry by entry against the same call over one entry at a time (which
the parity tests compare with the oracle). Every value comes from the same
operations on the same inputs, so equality is exact."""
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


def _run(P, n, cam, spl, act, g2, G, accumulate, n_sets, act_flags, mask_loss):
    s = [dict(ax=torch.full((n,), 0.5, device=DEV), ar=torch.full((n,), 0.25, device=DEV),
              cnt=torch.full((n,), 3, dtype=torch.int32, device=DEV),
              mr=torch.full((n,), 5, dtype=torch.int32, device=DEV) if k else None) for k in range(n_sets)]
    sets = [lib.grad_stats(x["ax"], x["ar"], x["cnt"], x["mr"]) for x in s]
    na = torch.tensor([act.numel()], dtype=torch.int32, device=DEV)
    lib.gs_project_bwd_ex(P, n, 3, act_flags, cam, spl, act if act.numel() else torch.zeros(1, dtype=torch.int32, device=DEV),
                          na, g2, G, accumulate, sets, mask_loss)
    return [t for x in s for t in (x["ax"], x["ar"], x["cnt"], x["mr"]) if t is not None]


@pytest.mark.parametrize("m", [0, 1, 31, 32, 33, 127, 128, 700])
@pytest.mark.parametrize("accumulate,n_sets,flags,mask_loss", [(False, 2, 0, 0.0), (True, 1, 0, 0.0),
                                                               (False, 0, lib.GS_VOLUME_MASK, 0.01),
                                                               (True, 2, lib.GS_VOLUME_MASK | lib.GS_OPACITY_ABS, 0.01)])
def test_list_lengths(m, accumulate, n_sets, flags, mask_loss):
    n = 800
    P = torch.zeros((n, 64))
    P[:, :59] = torch.from_numpy(synth.gaussians_uniform(n, 3)).float()
    P[:, :3] *= 3.0  # a good part lies outside the view
    P[:, 59] = torch.linspace(-6, 6, n)
    P = P.to(DEV)
    cam = lib.camera(synth.circle_cameras(8, 4.0, 70, 50)[1])
    spl = torch.zeros((n, 12), device=DEV)
    lib.gs_project_ex(P, n, 3, flags, cam, spl)
    seen = spl.view(torch.int32)[:, 10] > 0
    assert 0.1 < seen.float().mean() < 0.9
    g = torch.Generator().manual_seed(m)
    act = torch.randperm(n, generator=g)[:m].sort().values.to(torch.int32).to(DEV)
    rows = torch.randn((n, 12), generator=g).to(DEV)
    rows[:, 9:] = 0
    rows[~seen] = 0
    G0 = torch.randn((n, 64), generator=g).to(DEV)
    G, g2 = G0.clone(), rows.clone()
    stats = _run(P, n, cam, spl, act, g2, G, accumulate, n_sets, flags, mask_loss)
    Gr, g2r = G0.clone(), rows.clone()
    ref = None
    for e in act[:: max(1, m // 40)]:  # one entry at a time, up to about 40 of them
        st = _run(P, n, cam, spl, e.view(1), g2r, Gr, accumulate, n_sets, flags, mask_loss)
        k = int(e)
        assert torch.equal(G[k], Gr[k]), k
        assert not g2[k].any() and not g2r[k].any()
        for a, b in zip(stats, st):
            assert a[k] == b[k]
    listed = torch.zeros(n, dtype=torch.bool, device=DEV)
    listed[act.long()] = True
    assert torch.equal(G[~listed], G0[~listed]) and torch.equal(g2[~listed], rows[~listed])
    touched = listed & seen
    assert not g2[touched].any()
    for a in stats:  # what was not listed or not seen keeps its statistics
        assert (a[~touched] == a[~touched][0]).all()
    if not accumulate and m and not flags:
        assert not G[listed & ~seen].any()
    assert lib.gs_get_device_error() == 0
