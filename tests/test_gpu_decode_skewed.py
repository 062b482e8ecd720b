"""The decode step over batches in which one request is much longer than the others, over clusters of every size that the rule
for them takes, and at the edges of the rule (256 rows, one and a half times the mean)."""
import pytest

from tests.test_gpu_decode import run_and_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kept,H,Hkv", [
    ([256, 1, 1], 28, 4), ([257, 1, 0, 3], 28, 4), ([300, 100], 9, 1), ([301, 100, 100], 16, 1),
    ([9000] + [20] * 7, 8, 2), ([4000] + [33] * 60, 8, 4), ([70] * 50 + [2500], 16, 1), ([3000] + [0] * 30 + [17], 4, 2),
    ([600] * 30 + [900] * 30, 4, 2), ([500, 200, 200, 200], 4, 4),
])
def test_long_requests_among_short_ones(kept, H, Hkv):
    run_and_check(kept, H, Hkv, 128, "bf16", seed=len(kept) + max(kept))
