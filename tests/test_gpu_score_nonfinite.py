"""What a NaN reaches in the scores that are formed in one cluster launch: a key's every row that sees it, a row's every key that
it sees, and nothing else."""
import pytest
import torch

from paper_2510_25600_b200 import inputs
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


def _scores(dtype, d, length, window, obs, pool, spoil=None):
    batch = inputs.make_batch([0], [0], [length], 2, 2)
    wl = inputs.Workload("t", 5, dtype, 4, 2, d, 1, (0,), (0,), batch, inputs.STMask(2, 2), window, 0.5)
    x = inputs.make_qkv(wl, 0, "qk")
    q, k = gc.upload(x, "q", dtype), gc.upload(x, "k", dtype)
    if spoil:
        spoil(q, k)
    return gc.pk().purekv_lowlayer_score_ex(q, k, gc.device_batch(wl), window, obs, pool)


@pytest.mark.parametrize("length,at", [(60, 3), (300, 70), (300, 299), (1024, 1000), (1024, 5)])
def test_a_nan_key_reaches_all_scores_of_its_head(length, at):
    def spoil(q, k):
        k[at, 1, 2] = float("nan")

    base, got = _scores("fp32", 64, length, 16, 16, 1), _scores("fp32", 64, length, 16, 16, 1, spoil)
    assert torch.equal(got[0], base[0])
    # the last key is seen by the last row alone, which is enough
    assert got[1, :length - 16].isnan().all() and (got[1, length - 16:] == 0).all()


@pytest.mark.parametrize("dtype,d,length,row,pool", [("fp32", 64, 300, 40, 1), ("fp32", 64, 500, 70, 5), ("bf16", 64, 500, 200, 1),
                                                     ("bf16", 128, 900, 300, 7)])
def test_a_nan_row_reaches_the_keys_it_sees(dtype, d, length, row, pool):
    def spoil(q, k):
        q[row, 1, 2] = float("nan")

    base, got = _scores(dtype, d, length, 16, -1, pool), _scores(dtype, d, length, 16, -1, pool, spoil)
    assert torch.equal(got[1], base[1])  # heads 2 and 3
    reach = row + 1 + pool // 2
    assert got[0, :reach].isnan().all() and torch.equal(got[0, reach:], base[0, reach:])
