"""The decode step at the edges of its launch rule (one CTA, clusters of 2-16, one or three stages, four or eight warps)
and of its tiles (16-row trips, shares that leave CTAs of a cluster empty)."""
import pytest

from tests.test_gpu_decode import run_and_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kept,H,Hkv", [
    ([128], 28, 4), ([129], 28, 4),          # one trip of eight warps; the first cluster
    ([1, 130, 17, 2049], 16, 1),             # clusters of 16, most of whose CTAs have no row; G = 16
    ([257, 0, 31], 9, 1),                    # G = 9: the second row group holds one head
    ([64] * 40, 8, 4), ([65] * 40, 8, 4),    # four warps, one and three stages
    ([2100] * 75, 4, 2),                     # more CTAs than SMs, long shares: eight warps
])
def test_decode_launch_rule_edges(kept, H, Hkv):
    run_and_check(kept, H, Hkv, 128, "bf16", seed=len(kept) + max(kept))
