"""One-pass scores over 1 to 29 blocks of stacked window rows: the two groups of warps take turns with the blocks and share the
rows' log-sum-exp through two buffers each, so odd and even counts, a last block of few rows and a group without a block count."""
import pytest
import torch

from oracle import purekv_oracle as po
from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,window", [(1, 1, 128), (2, 2, 136), (2, 1, 128), (3, 1, 88), (4, 2, 256), (7, 1, 72), (7, 1, 520), (5, 1, 104)])
def test_scores_over_many_blocks_of_rows(H, Hkv, window):
    P = gc.pk()
    batch = inputs.make_batch([8, 0], [14, 2], [33, 200], 6, 7)  # 629 and 284 tokens
    if window > 284:
        batch = inputs.make_batch([8], [14], [33], 6, 7)
    wl = inputs.Workload("t", 11, "bf16", H, Hkv, 128, 1, (0,), (0,), batch, inputs.STMask(6, 7, tile=64), window, 0.5)
    x = inputs.make_qkv(wl, 0)
    db = gc.device_batch(wl)
    q, k, v = (gc.upload(x, n, "bf16") for n in "qkv")
    plan = P.purekv_plan_build(db, P.st_params(inputs.STMask(6, 7, tile=64, dense_causal=True)), P.BF16, 128, H, Hkv)
    lse = torch.empty((H, db.total_tokens), dtype=torch.float32, device="cuda")
    P.purekv_st_sparse_prefill(q, k, v, db, plan, lse=lse)
    c = torch.full((Hkv, db.total_tokens), float("nan"), dtype=torch.float32, device="cuda")
    P.purekv_lowlayer_score_lse(q, k, lse, db, window, c_out=c)
    ref = po.lowlayer_score(x["q"], x["k"], batch.cu_seqlens, window)
    assert gc.score_error(c.cpu().numpy(), ref) <= gc.SCORE_RTOL
