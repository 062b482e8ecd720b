"""Two waves and more of segments with rows of 256 bytes are selected without a workspace, with the indices and rows that the calls
with one give; fewer segments, other rows and segments too long for shared memory are refused as ever."""
import pytest
import torch

from paper_2510_25600_b200 import inputs  # noqa: F401  (the package's import checks the library)
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


def _call(P, name, c, k, v, db, bud, ws):
    idx = torch.full((v.shape[0], v.shape[2], bud.total_kept), -1, dtype=torch.int32, device="cuda")
    k_out, v_out = (torch.zeros((v.shape[0], bud.total_kept, *v.shape[2:]), dtype=v.dtype, device="cuda") for _ in range(2))
    b = P.C.byref(db.c)
    rest = (db.n_req and v.stride(0), v.shape[0], b, bud.window, bud.keep.data_ptr(), bud.h_keep.ctypes.data_as(P._i32p),
            bud.cu_kept.data_ptr(), bud.h_cu_kept.ctypes.data_as(P._i32p), v.shape[2], v.shape[3], P._dtype_code(v), idx.data_ptr(), None)
    tail = (None if ws is None else ws.data_ptr(), 0 if ws is None else ws.numel(), P._stream())
    if name == "topk":
        st = P._lib.purekv_select_topk(c.data_ptr(), v.data_ptr(), *rest, *tail)
    else:
        st = P._lib.purekv_select_compact(c.data_ptr(), k.data_ptr(), v.data_ptr(), *rest, k_out.data_ptr(), v_out.data_ptr(),
                                          k_out.stride(0), *tail)
    return st, idx, k_out, v_out


@pytest.mark.parametrize("dtype,d,hkv,layers,lens,taken", [
    ("bf16", 128, 4, 37, [300, 0, 41, 1000], True), ("bf16", 128, 4, 37, [700, 64], True), ("fp32", 64, 1, 296, [129], True),
    ("bf16", 128, 1, 296, [3], True), ("bf16", 128, 1, 295, [129], False), ("bf16", 64, 2, 200, [129], False),
])
def test_with_and_without(dtype, d, hkv, layers, lens, taken):
    P = gc.pk()
    db = P.Batch(lens, [0] * len(lens), [0] * len(lens))
    bud = P.Budget(db, 16, 0.4)
    g = torch.Generator(device="cuda").manual_seed(5)
    k, v = (torch.randn((layers, db.total_tokens, hkv, d), generator=g, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32)
            for _ in range(2))
    c = torch.rand((hkv, db.total_tokens), generator=g, device="cuda")
    ws = torch.empty(P.purekv_select_ws_bytes(db, layers, hkv), dtype=torch.uint8, device="cuda")
    for name in ("topk", "compact"):
        ref = _call(P, name, c, k, v, db, bud, ws)
        got = _call(P, name, c, k, v, db, bud, None)
        assert ref[0] == P.OK
        if taken:
            assert got[0] == P.OK and all(torch.equal(x, y) for x, y in zip(got[1:], ref[1:]))
        else:
            assert got[0] == P.ERR_WORKSPACE and (got[1] == -1).all()
