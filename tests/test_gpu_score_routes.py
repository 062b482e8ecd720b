"""Scores over the sizes at which the form changes: clusters in one wave and in several, 128 and 256 keys per CTA for the same
length, ragged batches, requests within their window (all, some), many blocks of rows; each against the oracle."""
import pytest

from oracle import purekv_oracle as po
from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,H,Hkv,lens,window,obs,pool", [
    ("bf16", 64, 8, 8, [2000], 40, 40, 1), ("bf16", 64, 8, 8, [1300, 90, 33], 64, 64, 1), ("bf16", 64, 4, 4, [600] * 9, 30, 30, 7),
    ("bf16", 64, 8, 8, [2100, 300], 130, 130, 1), ("bf16", 128, 2, 1, [50, 64, 9], 64, 64, 1), ("bf16", 128, 2, 1, [50, 0, 200], 64, 20, 5),
    ("bf16", 64, 14, 2, [300] * 40, 16, 16, 1), ("fp32", 64, 4, 2, [60, 33], 64, 64, 1), ("fp32", 64, 8, 8, [100, 260], 128, 128, 3),
    ("fp32", 64, 4, 4, [290] * 30, 200, 200, 1), ("fp32", 32, 8, 2, [1000] * 3, 60, 60, 1), ("fp32", 128, 7, 1, [280], 256, 256, 1),
])
def test_scores_where_the_form_changes(dtype, d, H, Hkv, lens, window, obs, pool):
    P = gc.pk()
    batch = inputs.make_batch([0] * len(lens), [0] * len(lens), lens, 2, 2)
    wl = inputs.Workload("t", 6, dtype, H, Hkv, d, 1, (0,), (0,), batch, inputs.STMask(2, 2), window, 0.5)
    x = inputs.make_qkv(wl, 0, "qk")
    q, k, db = gc.upload(x, "q", dtype), gc.upload(x, "k", dtype), gc.device_batch(wl)
    got = P.purekv_lowlayer_score_ex(q, k, db, window, obs, pool)
    ref = po.lowlayer_score_ex(x["q"], x["k"], batch.cu_seqlens, window, obs, pool)
    assert gc.score_error(got.cpu().numpy(), ref) <= gc.SCORE_RTOL
