"""Tiles of which a warp's 32 rows keep nothing, one, two, three or four of the 32-key chunks: the kernel reads only those that
are kept where there are two at most."""
import numpy as np
import pytest

from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


def _workload(heads, mask):
    batch = inputs.make_batch([5, 0], [7, 3], [90, 1], mask.grid_h, mask.grid_w)
    return inputs.Workload("chunks", 3, "bf16", heads, 1, 128, 1, (0,), (0,), batch, mask, 16, 0.25)


@pytest.mark.parametrize("tile", [64, 128])
@pytest.mark.parametrize("window", [1, 31, 32, 33, 64, 65, 97, 130])  # rows keep 1 .. 130 keys: 1-2, 2, 2-3 ... chunks of a tile
def test_local_windows_across_the_chunks(tile, window):
    wl = _workload(2, inputs.STMask(9, 11, anchor_frames=0, temporal_depth=0, spatial_radius=0, tile=tile, local_window=window))
    gc.check_prefill(wl, inputs.make_qkv(wl, 0))


@pytest.mark.parametrize("grid", [(8, 16), (12, 12), (10, 13), (16, 16)])  # the previous frame's cell: a diagonal, aligned and not
@pytest.mark.parametrize("heads", [2, 3])  # an odd group: two query tiles share a unit, each with chunks of its own
@pytest.mark.parametrize("scale", [1.0, 40.0])  # logits of several hundred: rows are redone against their maximum
def test_diagonals(grid, heads, scale):
    wl = _workload(heads, inputs.STMask(*grid, tile=128))
    x = inputs.make_qkv(wl, 0)
    x["q"], x["v"] = x["q"] * scale, x["v"] * 0.5  # (outputs below 4, where a step of bf16 is 2^-7)
    for n in "qv":
        x[n + "_bits"] = inputs.f32_to_bf16_bits(x[n])
        x[n] = inputs.bf16_bits_to_f32(x[n + "_bits"])
    gc.check_prefill(wl, x)
