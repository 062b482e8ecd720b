"""The plan's magic names its layout: plans with the kept halves behind the masks and byte-wide merge counters do not carry the
magic of those without, and the kernel refuses one that does."""
import numpy as np
import pytest
import torch

from paper_2510_25600_b200 import binding as pk, inputs

BEFORE = 0x504B5636  # no kept halves, merge counters of a word per head
MASK = inputs.STMask(8, 8, tile=128)


def _plan(device):
    batch = inputs.make_batch([20], [6], [40], 8, 8)
    b = pk.Batch(batch.seq_lens, batch.n_prefix, batch.n_frames, device=device)
    return b, *pk.purekv_plan_build_host(b, pk.st_params(MASK), pk.BF16, 128, 2, 1)


def test_the_magic_is_not_that_of_the_layout_before():
    _, plan, _ = _plan(None)
    assert pk.PlanHeaderView.from_buffer_copy(plan.tobytes()).magic != BEFORE


@pytest.mark.gpu
def test_a_plan_of_the_layout_before_is_refused():
    b, plan, info = _plan("cuda")
    plan = plan.copy()
    plan[:4] = np.frombuffer(np.uint32(BEFORE).tobytes(), dtype=np.uint8)
    t = b.total_tokens
    q, k, v = (torch.zeros((t, h, 128), dtype=torch.bfloat16, device="cuda") for h in (2, 1, 1))
    out = torch.full_like(q, 7.0)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    pk.purekv_st_sparse_prefill(q, k, v, b, pk.Plan(torch.from_numpy(plan).cuda(), info), out=out, status=status)
    # (read directly: the traceback of a raised error would keep the tensors alive past the test, until some later collection)
    assert status.item() == pk.ERR_BAD_PLAN and (out == 7.0).all()


@pytest.mark.parametrize("heads", [(1, 1), (2, 1), (7, 1), (28, 4)])
@pytest.mark.parametrize("frames,dense", [([0], False), ([3], False), ([16], False), ([16], True), ([5, 30, 1], False), ([40], True)])
@pytest.mark.parametrize("n_layers", [1, 2, 30])
def test_the_size_for_many_layers_is_enough_for_a_layer_at_a_time(heads, frames, dense, n_layers):
    batch = inputs.make_batch([5] * len(frames), frames, [40] * len(frames), 12, 13)
    b = pk.Batch(batch.seq_lens, batch.n_prefix, batch.n_frames, device=None)
    args = (b, pk.st_params(inputs.STMask(12, 13, tile=64, dense_causal=dense)), pk.BF16, 128, *heads)
    one, many = (pk.purekv_plan_build_host(*args, n_layers=n)[1].bytes_used for n in (1, n_layers))
    assert pk.purekv_plan_bytes(*args, n_layers=n_layers) == max(one, many) and pk.purekv_plan_bytes(*args) == one
