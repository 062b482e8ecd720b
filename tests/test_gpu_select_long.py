"""Few long segments, which 1024 threads each select from: keys in shared memory, one more than fit there, and many more (and one key less, which 512 threads do); distinct
scores and scores of which hundreds are equal.  The selection is the oracle's on the scores that the call itself reports."""
import numpy as np
import pytest
import torch

from oracle import purekv_oracle as po
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [[8191], [8192, 30], [51200], [51201], [300, 60001]], ids=str)
@pytest.mark.parametrize("distinct", [True, False])
def test_long_segments(lens, distinct):
    P = gc.pk()
    db = P.Batch(lens, [0] * len(lens), [0] * len(lens))
    bud = P.Budget(db, 48, 0.3)
    t, layers, hkv = db.total_tokens, 2, 2
    g = torch.Generator(device="cuda").manual_seed(len(lens) + t)
    v = torch.randn((layers, t, hkv, 128), generator=g, device="cuda").bfloat16() if distinct else torch.ones((layers, t, hkv, 128), device="cuda").bfloat16()
    c = torch.rand((hkv, t), generator=g, device="cuda")
    if not distinct:
        c = (c * 100).floor()
    s = torch.empty((layers, hkv, t), device="cuda")
    idx = P.purekv_select_topk(c, v, db, bud, s_out=s)
    assert torch.equal(idx, P.purekv_select_topk(c, v, db, bud))
    cu = np.concatenate([[0], np.cumsum(lens)])
    for layer in range(layers):
        ref, _ = po.select(s[layer].cpu().numpy().astype(np.float64), cu, 48, bud.h_keep, bud.h_cu_kept)
        assert np.array_equal(idx[layer].cpu().numpy(), ref)
