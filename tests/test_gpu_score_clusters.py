"""Scores in one cluster launch at the edges of its range: requests that end inside, at and behind a CTA's keys, clusters of 1
to 16, blocks of rows with absent rows, several row blocks, observations longer than the window, pools that reach into the
neighbouring CTAs; and the sizes just past the range, which the separate kernels take."""
import pytest

from oracle import purekv_oracle as po
from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,H,Hkv,lens,window,obs,pool", [
    ("bf16", 128, 8, 2, [1, 127, 128, 129, 300], 16, 16, 1), ("bf16", 64, 7, 1, [2048, 40], 64, 64, 1),
    ("bf16", 128, 4, 2, [2049, 0, 700], 50, 32, 7), ("bf16", 128, 4, 4, [4096], 100, 100, 129),
    ("bf16", 128, 4, 4, [4097], 100, 100, 7), ("bf16", 32, 16, 1, [500, 130], 8, 130, 5), ("bf16", 128, 4, 2, [260], 8, 600, 131),
    ("fp32", 64, 2, 1, [1, 64, 65, 288], 16, 16, 1), ("fp32", 256, 4, 2, [1024, 3], 33, 40, 63),
    ("fp32", 64, 4, 1, [1025], 16, 16, 7), ("fp32", 20, 4, 2, [150], 7, 90, 65),
])
def test_cluster_scores_match_the_oracle(dtype, d, H, Hkv, lens, window, obs, pool):
    P = gc.pk()
    batch = inputs.make_batch([0] * len(lens), [0] * len(lens), lens, 2, 2)
    wl = inputs.Workload("t", 5, dtype, H, Hkv, d, 1, (0,), (0,), batch, inputs.STMask(2, 2), window, 0.5)
    x = inputs.make_qkv(wl, 0, "qk")
    got = P.purekv_lowlayer_score_ex(gc.upload(x, "q", dtype), gc.upload(x, "k", dtype), gc.device_batch(wl), window, obs, pool)
    ref = po.lowlayer_score_ex(x["q"], x["k"], batch.cu_seqlens, window, obs, pool)
    assert gc.score_error(got.cpu().numpy(), ref) <= gc.SCORE_RTOL
