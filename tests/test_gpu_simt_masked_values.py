"""The CUDA-core prefill puts several key tiles of the plan into one chunk.  A row that keeps nothing of a tile takes nothing from
it, whatever stands there: an infinity or a NaN in its V or K leaves the row as it is without."""
import pytest
import torch

from oracle import purekv_oracle as po
from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu
GH, GW = 6, 7


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("dtype,d,tile,variant", [("fp32", 64, 16, "st"), ("fp32", 64, 32, "spatial"), ("bf16", 64, 16, "local"),
                                                  ("fp32", 256, 64, "st"), ("fp32", 128, 64, "spatial"), ("bf16", 128, 32, "st")])
def test_rows_that_keep_nothing_of_a_tile(dtype, d, tile, variant, value):
    P = gc.pk()
    batch = inputs.make_batch([9], [7], [40], GH, GW)
    mask = inputs.mask_variant(variant, GH, GW, tile=tile, local_window=40)
    wl = inputs.Workload("t", 5, dtype, 2, 1, d, 1, (0,), (0,), batch, mask, 16, 0.3)
    x = inputs.make_qkv(wl, 0)
    q, k, v = (gc.upload(x, n, dtype) for n in "qkv")
    db = gc.device_batch(wl)
    plan = P.purekv_plan_build(db, P.st_params(mask), P.BF16 if dtype == "bf16" else P.FP32, d, 2, 1)
    keeps = torch.from_numpy(po.mask_matrix(po.mask_params(mask), batch.seq_lens[0], 9, 7)).cuda()
    base = P.purekv_st_sparse_prefill(q, k, v, db, plan)
    spared = 0
    for j in (60, 101, 150, 230, 310):
        free = ~keeps[:, j // tile * tile:(j // tile + 1) * tile].any(dim=1)
        for t in (k, v):
            was = t[j].clone()
            t[j, 0, 3] = value
            err = (P.purekv_st_sparse_prefill(q, k, v, db, plan)[free].float() - base[free].float()).abs().max() if free.any() else 0.0
            assert err <= gc.ATTN_TOL[dtype]  # (such rows are formed anew, in another order)
            t[j] = was
        spared += int(free.sum())
    assert spared > 0
