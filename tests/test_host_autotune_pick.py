"""The autotuner's choice among launch shapes whose times differ by noise: the
smallest batch within 5% of the fastest, and the fastest of those."""
import pytest

from paper_2504_06716_gb300.autotune import pick


@pytest.mark.parametrize("times,want", [
    ({(1, 32): 1.02, (1, 64): 1.0, (2, 32): 1.01, (2, 256): 0.99}, (2, 32)),
    ({(1, 32): 1.2, (2, 64): 1.0, (2, 256): 0.98}, (2, 64)),
    ({(1, 32): 2.0, (2, 256): 1.0}, (2, 256)),
    ({(4, 128): 1.0}, (4, 128)),
])
def test_pick(times, want):
    assert pick(times) == want
