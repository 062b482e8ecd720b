"""V-norm scores at the edges of a warp's 16-row blocks: fewer rows than a block, a partly filled last block per layer, fewer
blocks than warps, layers that start inside a CTA's run, rows of 256 bytes in both types and other row lengths; with few
segments and with more than a wave of them, and compaction behind either."""
import numpy as np
import pytest
import torch

from oracle import purekv_oracle as po
from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,hkv,layers,lens", [
    ("bf16", 128, 1, 1, [1]), ("bf16", 128, 1, 5, [15]), ("bf16", 128, 3, 7, [16, 1]), ("bf16", 128, 2, 40, [17, 3, 64]),
    ("bf16", 128, 4, 3, [2500, 0, 733]), ("fp32", 64, 2, 9, [129, 31]), ("fp32", 64, 1, 160, [50]),
    ("bf16", 128, 2, 3, [1017, 1019]), ("bf16", 128, 1, 2, [1030]),  # 1017 kept rows of two requests (gathered), 515 of one (compacted)
    ("bf16", 64, 2, 3, [77, 5]), ("fp32", 20, 3, 2, [301]), ("bf16", 256, 1, 2, [40]),
])
def test_scores_selection_and_rows(dtype, d, hkv, layers, lens):
    P = gc.pk()
    batch = inputs.make_batch([0] * len(lens), [0] * len(lens), lens, 2, 2)
    wl = inputs.Workload("t", 9, dtype, hkv, hkv, d, layers, (0,), (0,), batch, inputs.STMask(2, 2), 4, 0.5)
    db = gc.device_batch(wl)
    bud = P.Budget(db, 4, 0.5)
    rng = np.random.default_rng(7)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    t = db.total_tokens
    k, v = (torch.from_numpy(rng.standard_normal((layers, t, hkv, d), dtype=np.float32)).to(tdt).cuda() for _ in range(2))
    c = torch.from_numpy(rng.random((hkv, t), dtype=np.float32)).cuda()
    s = torch.full((layers, hkv, t), -1.0, dtype=torch.float32, device="cuda")
    idx = P.purekv_select_topk(c, v, db, bud, s_out=s)
    kc, vc = P.purekv_compact_kv(k, v, idx, db, bud)
    both = P.purekv_select_compact(c, k, v, db, bud)
    ref = c.double()[None] * v.double().norm(dim=3).permute(0, 2, 1)
    # d squares summed in fp32 in any order: at most (d + 1) roundings, halved by the root, and one each for root and product
    assert ((s.double() - ref).abs() <= ((d + 1) / 2 + 2) * 2.0 ** -24 * ref).all()
    h_keep, cu_kept = po.budgets(batch.seq_lens, 4, 0.5)
    s_h, idx_h = s.double().cpu().numpy(), idx.cpu().numpy()
    for l in range(layers):
        assert np.array_equal(po.select(s_h[l], batch.cu_seqlens, 4, h_keep, cu_kept)[0], idx_h[l])
    first = torch.from_numpy(np.repeat(np.asarray(batch.cu_seqlens[:-1]), np.diff(cu_kept))).cuda()
    rows = (idx.long() + first).permute(0, 2, 1)[..., None].expand(-1, -1, -1, d)
    assert torch.equal(kc, k.gather(1, rows)) and torch.equal(vc, v.gather(1, rows))
    assert torch.equal(both[0], idx) and torch.equal(both[1], kc) and torch.equal(both[2], vc)
