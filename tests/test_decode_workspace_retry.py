"""purekv_decode_attention's own workspace: sized for the requests of the call, not for all of the budget's, and asked for once."""
import types

import numpy as np
import pytest
import torch

from paper_2510_25600_b200 import binding as P
from tests.gpu_common import ATTN_TOL

# the split is not monotone in the longest request: 4736 rows are cut finer than 4737
KEPT = [4736, 4737]


def _budget(device="cpu"):
    cu = np.concatenate([[0], np.cumsum(KEPT)]).astype(np.int32)
    return types.SimpleNamespace(h_cu_kept=cu, cu_kept=torch.from_numpy(cu.copy()).to(device))


@pytest.mark.parametrize("answers,raises", [([P.ERR_WORKSPACE, P.OK], False), ([P.ERR_WORKSPACE] * 2, True), ([P.ERR_INVALID_ARG], True)])
def test_one_retry_with_what_the_call_needs(monkeypatch, answers, raises):
    given = []

    def native(*args):
        given.append(args[14])
        return answers[len(given) - 1]

    monkeypatch.setattr(P, "_marshal", types.SimpleNamespace(purekv_decode_attention=native))
    monkeypatch.setattr(P, "_stream", lambda: 0)
    q, rows = torch.zeros((1, 4, 64)), torch.zeros((sum(KEPT), 4, 64))
    if raises:
        with pytest.raises(P.PureKVError):
            P.purekv_decode_attention(q, rows, rows, _budget())
    else:
        P.purekv_decode_attention(q, rows, rows, _budget())
    need = [P.purekv_decode_ws_bytes(1, n, 4, 4, 64) for n in KEPT]
    assert need[0] > need[1] and given == [0, need[0]][:len(answers)]


@pytest.mark.gpu
def test_the_first_request_alone():
    g = torch.Generator(device="cuda").manual_seed(2)
    rows = [torch.randn((sum(KEPT), 4, 64), generator=g, device="cuda") for _ in range(2)]
    q = torch.randn((1, 4, 64), generator=g, device="cuda")
    got = P.purekv_decode_attention(q, *rows, _budget("cuda"))
    k, v = (x[:KEPT[0]].double() for x in rows)
    ref = torch.einsum("hj,jhd->hd", (torch.einsum("hd,jhd->hj", q[0].double(), k) / 8.0).softmax(1), v)
    assert (got[0].double() - ref).abs().max() <= ATTN_TOL["fp32"]
