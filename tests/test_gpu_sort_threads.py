"""gs_sort called from two host threads at once, each on its own stream and
buffers: calls on different streams are independent as long as their buffers
are, so every list equals the one a single thread gets, word for word. The
grids differ in the shared memory their passes ask for: depth passes of nine
bits, super-tile passes of a few bits, and the one-block sort of few Gaussians."""
import threading

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


class _Sorter:
    """One view's projected splats, and buffers to sort them into."""

    def __init__(self, n, width, height, tile, seed):
        scene = synth.surface_scene(n, n, 1, width, height, seed=seed)
        self.n, self.cam, self.cap = n, lib.camera(scene.cameras[0], tile=tile), 24 * n + 20000
        P = torch.zeros((n, lib.ROW), device=DEV)
        P[:, :59] = torch.from_numpy(scene.init).to(DEV)
        self.splats = torch.zeros((n, lib.SPLAT), device=DEV)
        lib.gs_project(P, n, 3, self.cam, self.splats)
        self.ws = torch.zeros(lib.gs_sort_workspace_bytes(n, self.cap, self.cam), dtype=torch.uint8, device=DEV)
        self.vals = torch.zeros(self.cap, dtype=torch.int32, device=DEV)
        self.ranges = torch.zeros((self.cam.tiles, 2), dtype=torch.int32, device=DEV)
        self.count = torch.zeros(1, dtype=torch.int64, device=DEV)

    def sort(self, stream=None):
        lib.gs_sort(self.splats, self.n, self.cam, self.ws, self.cap, self.vals, self.ranges, self.count, stream)

    def lists(self):
        torch.cuda.synchronize()
        k = int(self.count.item())
        assert 0 < k <= self.cap
        return self.vals[:k].clone(), self.ranges.clone(), k


@pytest.mark.parametrize("first,second", [((20011, 400, 300, 16), (30001, 1001, 667, 8)),
                                          ((5000, 300, 200, 16), (40000, 640, 480, 8))])
def test_sorts_of_two_threads(first, second):
    sorters = [_Sorter(*first, 1), _Sorter(*second, 2)]
    want = []
    for s in sorters:
        s.sort()
        want.append(s.lists())
        s.vals.fill_(-1)
        s.ranges.fill_(-1)
    torch.cuda.synchronize()
    start, failed = threading.Barrier(2), []

    def work(s):
        try:
            stream = torch.cuda.Stream()
            start.wait(60)
            for _ in range(300):
                s.sort(stream)
            stream.synchronize()
        except Exception as e:  # a thread's failure is the test's
            failed.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in sorters]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for s, (vals, ranges, k) in zip(sorters, want):
        got = s.lists()
        assert got[2] == k and torch.equal(got[0], vals) and torch.equal(got[1], ranges)
    assert lib.gs_get_device_error() == 0
