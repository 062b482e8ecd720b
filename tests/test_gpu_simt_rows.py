"""The CUDA-core prefill over its forms: rows per CTA (8, 16, 32, 64 by the job's size), key tiles shorter and longer than a
chunk, query tiles with few valid rows, lists that end in the middle of a chunk."""
import pytest

from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,H,Hkv,tile,frames", [
    ("fp32", 64, 2, 1, 16, 3), ("fp32", 32, 2, 1, 16, 1), ("fp32", 64, 7, 1, 32, 3), ("fp32", 128, 32, 8, 32, 3),
    ("fp32", 64, 40, 8, 64, 6), ("bf16", 64, 40, 8, 128, 6), ("fp32", 256, 4, 2, 128, 2), ("bf16", 256, 32, 8, 64, 4),
])
def test_forms_match_the_oracle(dtype, d, H, Hkv, tile, frames):
    batch = inputs.make_batch([3, 0], [frames, 1], [14, 1], 9, 11)
    wl = inputs.Workload("t", 7, dtype, H, Hkv, d, 1, (0,), (0,), batch, inputs.STMask(9, 11, tile=tile), 16, 0.25)
    gc.check_prefill(wl, inputs.make_qkv(wl, 0))
