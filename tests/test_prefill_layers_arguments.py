"""Strides between layers that no launch could take are refused before the first layer is launched (here, without a GPU, a launch
would come back as PUREKV_ERR_CUDA)."""
import ctypes as C

import numpy as np
import pytest

from paper_2510_25600_b200 import binding as P
from paper_2510_25600_b200 import inputs


@pytest.mark.parametrize("dtype,d,tile,n_layers", [(P.BF16, 128, 64, 8), (P.BF16, 128, 64, 1), (P.FP32, 64, 16, 1)])
@pytest.mark.parametrize("which,by", [("q", 1), ("kv", 1), ("o", 1), ("o", 8)])
def test_a_stride_that_misaligns_the_second_layer(dtype, d, tile, n_layers, which, by):
    if by == 8 and dtype == P.FP32:
        by = 2  # (8 bytes; 8 bf16 are 16 bytes, which the tensor-core kernel's O does not take)
    batch = inputs.make_batch([3], [9], [20], 8, 8)
    b = P.Batch(batch.seq_lens, batch.n_prefix, batch.n_frames, device=None)
    buf, info = P.purekv_plan_build_host(b, P.st_params(inputs.STMask(8, 8, tile=tile)), dtype, d, 2, 1, n_layers=n_layers)
    t = b.total_tokens
    strides = {"q": t * 2 * d, "kv": t * d, "o": t * 2 * d}
    strides[which] += by
    room = np.zeros(64, dtype=np.uint8)
    a = (room.ctypes.data + 31) & ~31
    st = P._lib.purekv_st_sparse_prefill_layers(a, a, a, a, None, strides["q"], strides["kv"], strides["o"], 0, 2, C.byref(b.c), a,
                                                C.byref(info), 2, 1, d, dtype, 0.0, a, info.ws_bytes, None, None)
    assert st == P.ERR_INVALID_ARG
