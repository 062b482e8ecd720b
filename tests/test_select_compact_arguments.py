"""purekv_select_compact takes and refuses the same calls whichever of its two routes the job's size sends it to."""
import subprocess
import sys

import pytest
import torch

from tests.test_host_library import ROOT

NEGATIVE = """
import ctypes as C
import numpy as np
from paper_2510_25600_b200 import binding as P
cu = np.zeros(4, dtype=np.int32)
p = cu.ctypes.data_as(C.POINTER(C.c_int32))
b = P.CBatch(-(1 << 28), 0, None, p, p, p)
a = 1 << 20
st = P._lib.purekv_select_compact(a, a, a, 0, 1, C.byref(b), 16, a, p, a, p, 1, 128, P.BF16, a, None, a, a, 0, None, 0, None)
assert st == P.ERR_INVALID_ARG, st
"""


def test_a_negative_request_count_is_refused_before_anything_is_read():
    subprocess.run([sys.executable, "-c", NEGATIVE], cwd=ROOT, check=True, timeout=120)


@pytest.mark.gpu
@pytest.mark.parametrize("lens,layers", [([2700], 3), ([1100, 2000], 2), ([40, 9], 160)])
def test_layers_may_share_their_rows(lens, layers):
    from tests import gpu_common as gc
    P = gc.pk()
    db = P.Batch(lens, [0] * len(lens), [0] * len(lens))
    bud = P.Budget(db, 16, 0.5)
    g = torch.Generator(device="cuda").manual_seed(3)
    rows = [torch.randn((1, db.total_tokens, 2, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
    c = torch.rand((2, db.total_tokens), generator=g, device="cuda")
    ref = P.purekv_select_compact(c, *(x.repeat(layers, 1, 1, 1) for x in rows), db, bud)
    got = P.purekv_select_compact(c, *(x.expand(layers, -1, -1, -1) for x in rows), db, bud)
    assert all(torch.equal(x, y) for x, y in zip(got, ref))
