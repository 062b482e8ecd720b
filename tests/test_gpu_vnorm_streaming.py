"""Selection from a V that is larger than what the L2 keeps (its loads are marked as the first to be evicted) and from one just
below: the scores against 64 bits, the indices against the oracle's rule on those scores."""
import numpy as np
import pytest
import torch

from oracle import purekv_oracle as po
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens,layers", [(8191, 12), (8193, 12), (3001, 40)])  # 96 MiB is 12 layers of 8192 tokens x 4 heads
def test_scores_and_selection(tokens, layers):
    P = gc.pk()
    db = P.Batch([tokens], [0], [0])
    bud = P.Budget(db, 32, 0.1)
    g = torch.Generator(device="cuda").manual_seed(4)
    v = torch.randn((layers, tokens, 4, 128), generator=g, device="cuda").to(torch.bfloat16)
    c = torch.rand((4, tokens), generator=g, device="cuda")
    s = torch.full((layers, 4, tokens), -1.0, device="cuda")
    idx = P.purekv_select_topk(c, v, db, bud, s_out=s)
    h_keep, cu_kept = po.budgets([tokens], 32, 0.1)
    cu = np.array([0, tokens], dtype=np.int32)
    for l in (0, layers // 2, layers - 1):
        ref = c.double() * v[l].double().norm(dim=2).T
        # 128 squares summed in fp32 in any order: at most 129 roundings, halved by the root, and one each for root and product
        assert ((s[l].double() - ref).abs() <= (129 / 2 + 2) * 2.0 ** -24 * ref).all()
        assert np.array_equal(po.select(s[l].double().cpu().numpy(), cu, 32, h_keep, cu_kept)[0], idx[l].cpu().numpy())
