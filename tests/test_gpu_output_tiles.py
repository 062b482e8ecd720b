"""Whole query tiles leave through shared memory and the copy engine, cut ones row by row: requests whose last tile is whole,
short of it and just beyond, one behind the other, so that a row too many would land in the next request."""
import pytest

from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [(1, 1), (2, 1), (3, 1), (6, 2)])  # one slot, both, twin units (whole with whole, whole with cut)
@pytest.mark.parametrize("dense", [False, True])
def test_tiles_whole_and_cut(heads, dense):
    lens = [128, 127, 256, 129, 1, 255, 384, 257]
    batch = inputs.make_batch([0] * 8, [1] * 8, [length - 1 for length in lens], 1, 1)
    assert list(batch.seq_lens) == lens
    wl = inputs.Workload("tiles", 3, "bf16", *heads, 128, 1, (0,), (0,), batch, inputs.STMask(1, 1, tile=64, dense_causal=dense), 16, 0.25)
    x = inputs.make_qkv(wl, 0)
    gc.check_prefill(wl, x)             # a unit per CTA at most
    gc.check_prefill(wl, x, n_ctas=2)   # many: a stage is staged again and again
