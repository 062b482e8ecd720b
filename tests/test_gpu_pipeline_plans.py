"""After a pass whose layers are all dense the sparse mask's plan is there for who asks for it, and a layer can be run with it."""
import pytest
import torch

from oracle import purekv_oracle as po
from paper_2510_25600_b200 import inputs
from paper_2510_25600_b200.pipeline import PureKVPipeline
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,tile", [("fp32", 64, 16), ("bf16", 128, 64)])
def test_the_sparse_plan_of_a_pass_without_sparse_layers(dtype, d, tile):
    batch = inputs.make_batch([10], [5], [20], 8, 8)
    mask = inputs.STMask(8, 8, tile=tile)
    wl = inputs.Workload("t", 3, dtype, 2, 1, d, 1, (0,), (0,), batch, mask, 16, 0.3)
    x = inputs.make_qkv(wl, 0)
    q, k, v = (gc.upload(x, n, dtype)[None] for n in "qkv")
    pipe = PureKVPipeline(batch.seq_lens, batch.n_prefix, batch.n_frames, mask, 1, 2, 1, d, q.dtype, (0,), (0,), 16, 0.3)
    pipe.run_device(q, k, v)
    assert pipe.plan_st.info.n_qtiles > 0 and pipe.plan_st is pipe.plan_st
    out = torch.empty_like(q[0])
    gc.pk().purekv_st_sparse_prefill(q[0], k[0], v[0], pipe.batch, pipe.plan_st, out=out, ws=pipe.prefill_ws)
    ref, _ = po.prefill(x["q"], x["k"], x["v"], batch.cu_seqlens, batch.n_prefix, batch.n_frames, po.mask_params(mask))
    assert abs(gc.to_numpy_f32(out) - ref).max() <= gc.ATTN_TOL[dtype]
