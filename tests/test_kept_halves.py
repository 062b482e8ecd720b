"""The 64-key halves of a tile that hold any kept pair: the words behind the masks of a tensor-core plan say it for every entry
of the list, and the kernel that skips the others still computes the oracle's attention."""
import numpy as np
import pytest

from paper_2510_25600_b200 import binding as pk, inputs
from tests.test_host_library import parse_plan

# prefixes that cut frames across tiles, frames shorter and longer than a half, a last tile of less than a half, odd groups
CASES = [(1, 1, [64], [5], [70], 8, 8, 128), (3, 1, [20, 0], [6, 4], [40, 200], 9, 11, 128), (7, 1, [64], [4], [64], 16, 16, 128),
         (4, 2, [0], [3], [33], 24, 24, 128), (5, 1, [64, 5], [9, 1], [1, 90], 12, 12, 64)]


def _workload(H, Hkv, prefix, frames, text, gh, gw, tile):
    batch = inputs.make_batch(prefix, frames, text, gh, gw)
    return inputs.Workload("halves", 3, "bf16", H, Hkv, 128, 1, (0,), (0,), batch, inputs.STMask(gh, gw, tile=tile), 16, 0.25)


@pytest.mark.parametrize("case", CASES)
def test_plan_lists_the_kept_halves(case):
    wl = _workload(*case)
    b = pk.Batch(wl.batch.seq_lens, wl.batch.n_prefix, wl.batch.n_frames, device=None)
    buf, _ = pk.purekv_plan_build_host(b, pk.st_params(wl.mask), pk.BF16, 128, wl.n_q_heads, wl.n_kv_heads, 0)
    p = parse_plan(buf)
    ent, masks = p["entries"], p["masks"]
    halves = masks[len(masks) - len(ent):]
    for (x, at), h in zip(ent, halves):
        want = (x >> 2) & 3
        if x & 3 == 2:  # a bit mask: rows of four words, two to a half
            words = masks[at:at + 512].reshape(128, 2, 2)
            want &= int(words[:, 0].any()) | int(words[:, 1].any()) << 1
        assert h == want


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES)
def test_prefill_without_the_empty_halves(case):
    from tests import gpu_common as gc
    wl = _workload(*case)
    gc.check_prefill(wl, inputs.make_qkv(wl, 0))
