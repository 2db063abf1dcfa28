"""Statistics windows of the projection backward that share arrays, with one
another or within themselves: every addition counts, as if made one after
another (the increments, taken from a call with arrays of their own, are added
in that order in float32, so equality is exact)."""
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


# places of the eight arrays: (xyz, rgb, count, radius) of the first and of the second window
@pytest.mark.parametrize("places", ["abcd abcd", "abcd aefg", "abcd ebfg", "abcd efcg", "abcd efgd", "aacd efgh",
                                    "abcd bahg", "abcd efgh"])
@pytest.mark.parametrize("n", [1, 33, 700])
def test_every_addition_counts(n, places):
    P = torch.zeros((n, 64))
    P[:, :59] = torch.from_numpy(synth.gaussians_uniform(n, 3)).float()
    P = P.to(DEV)
    cam = lib.camera(synth.circle_cameras(8, 4.0, 70, 50)[1])
    spl = torch.zeros((n, 12), device=DEV)
    lib.gs_project(P, n, 3, cam, spl)
    radius = spl.view(torch.int32)[:, 10].clone()
    seen = radius > 0
    assert seen.any()
    g = torch.Generator().manual_seed(n)
    rows = torch.randn((n, 12), generator=g).to(DEV)
    rows[:, 9:] = 0
    rows[~seen] = 0
    act = torch.arange(n, dtype=torch.int32, device=DEV)
    na = torch.full((1,), n, dtype=torch.int32, device=DEV)

    def run(sets):
        G = torch.zeros((n, 64), device=DEV)
        lib.gs_project_bwd_stats(P, n, 3, cam, spl, act, na, rows.clone(), G, False, sets)
        return G

    inc = [torch.zeros(n, device=DEV), torch.zeros(n, device=DEV), torch.zeros(n, dtype=torch.int32, device=DEV)]
    G = run([lib.grad_stats(*inc)])
    first, second = places.split()
    arrays = {}
    for w in (first, second):
        for k, p in enumerate(w):
            if p not in arrays:
                arrays[p] = (torch.rand(n, generator=g) if k < 2
                             else torch.randint(0, 9, (n,), generator=g, dtype=torch.int32)).to(DEV)
    want = {p: t.clone() for p, t in arrays.items()}
    for w in (first, second):
        for k, p in enumerate(w):
            if k < 3:
                want[p] += torch.where(seen, inc[k], torch.zeros_like(inc[k]))
            else:
                want[p] = torch.where(seen, torch.maximum(want[p], radius), want[p])
    sets = [lib.grad_stats(*(arrays[p] for p in w)) for w in (first, second)]
    assert torch.equal(run(sets), G)
    for p, t in want.items():
        assert torch.equal(arrays[p], t), p
    assert lib.gs_get_device_error() == 0
