"""The autotuner times a launch shape's pixels per thread and not its batch,
which no kernel reads: one timing per pixels-per-thread, and the fastest of
them taken even where another is within a few percent."""
from paper_2504_06716_gb300 import autotune


def test_one_timing_per_pixels_per_thread(monkeypatch):
    timed = []

    def fake(fn, reps):
        fn()  # hands over the launch shape
        # were the four batches timed apart, noise of 3% would decide
        return {1: 1.03, 2: 1.0, 4: 1.4}[timed[-1][0]] * (1.0 if len(timed) % 2 else 1.03)

    monkeypatch.setattr(autotune, "_time", fake)
    times = autotune.time_shapes(lambda cfg: timed.append((cfg.pixels_per_thread, cfg.batch)), (2, 1, 4),
                                 (32, 64, 128, 256), 3)
    assert [p for p, _ in timed] == [2, 1, 4]
    assert set(times) == {(p, b) for p in (1, 2, 4) for b in (32, 64, 128, 256)}
    assert all(times[(p, b)] == times[(p, 32)] for p, b in times)
    assert autotune.pick(times) == (2, 32)
