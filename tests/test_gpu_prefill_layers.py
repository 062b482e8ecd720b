"""Several layers in one call: each layer comes out as its own call with the same plan gives it, and as the oracle computes it."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import purekv_oracle as po
from paper_2510_25600_b200 import binding as pk, inputs
from tests import gpu_common as gc

# heads / kv heads, prefix, frames, text, grid, skip, layers, dense: one tile and less, odd groups (twin units), last tiles cut by
# the layer's end (rows past it must not come from the next layer), requests of exactly one tile (units of one key tile in a row)
CASES = [(1, 1, [0], [1], [16], 5, 7, 128, 2, False), (3, 1, [20, 0], [6, 4], [40, 200], 9, 11, 64, 3, False),
         (4, 2, [0], [3], [33], 24, 24, 128, 5, True), (7, 1, [64], [4], [64], 16, 16, 128, 4, False),
         (3, 1, [0] * 6, [1] * 6, [112] * 6, 4, 4, 64, 4, False)]


def _case(H, Hkv, prefix, frames, text, gh, gw, tile, layers, dense):
    batch = inputs.make_batch(prefix, frames, text, gh, gw)
    return inputs.Workload("layers", 3, "bf16", H, Hkv, 128, layers, (0,), (0,), batch, inputs.STMask(gh, gw, tile=tile, dense_causal=dense),
                           16, 0.25)


def _plan(wl, device, n_layers, n_ctas=0):
    b = pk.Batch(wl.batch.seq_lens, wl.batch.n_prefix, wl.batch.n_frames, device=device)
    return b, *pk.purekv_plan_build_host(b, pk.st_params(wl.mask), pk.BF16, 128, wl.n_q_heads, wl.n_kv_heads, n_ctas=n_ctas,
                                         n_layers=n_layers)


@pytest.mark.parametrize("case", CASES)
def test_a_plan_for_many_layers_leaves_lists_whole(case):
    _, one, _ = _plan(_case(*case), None, 1)
    _, buf, info = _plan(_case(*case), None, 30)
    assert info.max_chunks == 1 and info.ws_bytes == 0 and info.n_units > 0
    old, new = (pk.PlanHeaderView.from_buffer_copy(x.tobytes()) for x in (one, buf))
    for f in ("magic", "n_qtiles", "n_ctas", "off_entries", "n_q_heads", "n_kv_heads"):
        assert getattr(old, f) == getattr(new, f)


def test_few_layers_of_a_long_list_keep_their_chunks():
    batch = inputs.make_batch([64], [80], [64], 16, 16)  # one head: 161 lists of up to 161 entries for 148 CTAs
    b = pk.Batch(batch.seq_lens, batch.n_prefix, batch.n_frames, device=None)
    params = pk.st_params(inputs.STMask(16, 16, tile=128, dense_causal=True))
    chunks = [pk.purekv_plan_build_host(b, params, pk.BF16, 128, 1, 1, n_layers=n)[1].max_chunks for n in (1, 2, 40)]
    assert chunks[0] == chunks[1] > 1 and chunks[2] == 1


@pytest.mark.gpu
@pytest.mark.parametrize("n_ctas", [0, 2, 5])  # a unit or two for each CTA; few CTAs, which go through the units of layer after layer
@pytest.mark.parametrize("case", CASES)
def test_layers_are_their_own_calls(case, n_ctas):
    wl = _case(*case)
    layers, t, pad = wl.n_layers, wl.batch.total_tokens, 3
    xs = [inputs.make_qkv(wl, n) for n in range(layers)]
    b, buf, info = _plan(wl, "cuda", 30, n_ctas)
    assert info.max_chunks == 1 and (n_ctas == 0 or info.n_ctas == n_ctas)
    assert n_ctas == 0 or info.n_units == 1 or info.n_units * layers >= 4 * n_ctas
    plan = pk.Plan(torch.from_numpy(buf.copy()).cuda(), info)
    stack = lambda n, width: torch.cat([torch.cat([gc.upload(x, n, "bf16"), torch.full((pad, width, 128), float("nan"), dtype=torch.bfloat16, device="cuda")])
                                        for x in xs]).view(layers, t + pad, width, 128)[:, :t]  # rows of NaN between the layers
    q, k, v = (stack(n, w) for n, w in (("q", wl.n_q_heads), ("k", wl.n_kv_heads), ("v", wl.n_kv_heads)))
    out = torch.full((layers, t + pad, wl.n_q_heads, 128), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((layers, wl.n_q_heads, t), 7.0, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        pk.purekv_st_sparse_prefill_layers(q, k, v, b, plan, out=out[:, :t], lse=lse, status=status)
    assert status.item() == 0 and (out[:, t:] == 7.0).all()
    assert _launches(lambda: pk.purekv_st_sparse_prefill_layers(q, k, v, b, plan, out=out[:, :t], lse=lse, status=status)) == 1
    for n in range(layers):
        one, one_lse = torch.empty_like(out[n, :t]), torch.empty_like(lse[n])
        pk.purekv_st_sparse_prefill(q[n], k[n], v[n], b, plan, out=one, lse=one_lse, status=status)
        assert torch.equal(one, out[n, :t]) and torch.equal(one_lse, lse[n])
    m = po.mask_params(wl.mask)
    ref, _ = po.prefill(xs[-1]["q"], xs[-1]["k"], xs[-1]["v"], wl.batch.cu_seqlens, wl.batch.n_prefix, wl.batch.n_frames, m)
    assert np.abs(gc.to_numpy_f32(out[-1, :t]) - ref).max() <= gc.ATTN_TOL["bf16"]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,n_layers,one_q", [("fp32", 3, True), ("fp32", 3, False), ("bf16", 1, False), ("bf16", 30, True)])
def test_layers_that_cannot_share_a_launch(dtype, n_layers, one_q):
    """The CUDA-core kernel; a plan with split lists; one Q for all layers (stride 0) under a plan with whole ones."""
    batch = inputs.make_batch([10], [12], [20], 8, 8)
    d = 64 if dtype == "fp32" else 128
    wl = inputs.Workload("l", 3, dtype, 2, 1, d, 3, (0,), (0,), batch, inputs.STMask(8, 8, tile=16 if dtype == "fp32" else 64), 16, 0.3)
    xs = [inputs.make_qkv(wl, n) for n in range(3)]
    q, k, v = (torch.stack([gc.upload(x, n, dtype) for x in xs]) for n in "qkv")
    if one_q:
        q = q[:1].expand(3, -1, -1, -1)
    b = pk.Batch(batch.seq_lens, batch.n_prefix, batch.n_frames)
    buf, info = pk.purekv_plan_build_host(b, pk.st_params(wl.mask), pk.BF16 if dtype == "bf16" else pk.FP32, d, 2, 1, n_layers=n_layers)
    assert dtype == "fp32" or (info.max_chunks > 1) == (n_layers == 1)
    plan = pk.Plan(torch.from_numpy(buf.copy()).cuda(), info)
    out = pk.purekv_st_sparse_prefill_layers(q, k, v, b, plan)
    ws, again = torch.empty(max(16, info.ws_bytes), dtype=torch.uint8, device="cuda"), torch.empty_like(out)
    assert _launches(lambda: pk.purekv_st_sparse_prefill_layers(q, k, v, b, plan, out=again, ws=ws)) == 3
    for n in range(3):
        assert torch.equal(out[n], pk.purekv_st_sparse_prefill(q[n], k[n], v[n], b, plan))


def _launches(call):
    """Kernels that `call` launches: the nodes of a graph that it is captured in."""
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        call()
    n = ctypes.c_size_t()
    assert ctypes.CDLL("libcuda.so.1").cuGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


def _pass(scored):
    from paper_2510_25600_b200.pipeline import PureKVPipeline
    batch = inputs.make_batch([10, 3], [12, 5], [20, 140], 12, 12)
    mask = inputs.STMask(12, 12, tile=64)
    wl = inputs.Workload("p", 3, "bf16", 4, 2, 128, 6, (0, 1), (2, 3, 4, 5), batch, mask, 16, 0.3)
    xs = [inputs.make_qkv(wl, n) for n in range(6)]
    q, k, v = (torch.stack([gc.upload(x, n, "bf16") for x in xs]) for n in "qkv")
    return PureKVPipeline(batch.seq_lens, batch.n_prefix, batch.n_frames, mask, 6, 4, 2, 128, q.dtype, scored, (2, 3, 4, 5), 16, 0.3), q, k, v


@pytest.mark.gpu
def test_a_pass_in_launches_of_many_layers_is_the_layers_one_by_one():
    pipe, q, k, v = _pass((0, 1))
    pipe.run_device(q, k, v)
    assert pipe.prefill_launches == 2 and pipe.plan_st.info.max_chunks == 1
    o, lse = pipe.o.clone(), pipe.lse.clone()
    pipe.o.fill_(float("nan"))
    pipe.lse.fill_(float("nan"))
    pipe.build_plans()  # for a layer at a time: lists are cut where that ends a launch sooner
    for n in range(6):
        pipe.prefill_layer(n, q[n], k[n], v[n])
    pipe.check_status()
    # either way of summing rounds P and the output to bf16: each is within the oracle's tolerance, the two within both
    assert (pipe.o.float() - o.float()).abs().max().item() <= 2 * gc.ATTN_TOL["bf16"]
    assert (pipe.lse - lse).abs().max().item() <= 2 * 2e-3


@pytest.mark.gpu
@pytest.mark.parametrize("scored", [(1,), (0, 1), (1, 0)], ids=str)
def test_the_dense_layers_share_a_launch_whichever_are_scored(scored):
    pipe, q, k, v = _pass(scored)
    whole, *_ = _pass((0, 1))
    for p in (pipe, whole):
        p.run_device(q, k, v)
        p.check_status()
        assert p.prefill_launches == 2
    assert torch.equal(pipe.o, whole.o) and pipe.lse.shape == (len(scored), 4, pipe.batch.total_tokens)
    for n, layer in enumerate(scored):
        assert torch.equal(pipe.lse[n], whole.lse[layer]) and torch.equal(pipe.c[n], whole.c[layer])


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["sequence", "one Q for all", "events"])
def test_layers_launched_one_by_one_are_planned_so(form):
    pipe, q, k, v = _pass((0, 1))
    if form == "one Q for all":
        q = q[:1].expand(6, -1, -1, -1)
    events = [[torch.cuda.Event() for _ in range(2)] for _ in range(6)] if form == "events" else None
    pipe.run_device(list(q) if form == "sequence" else q, k, v, events=events)
    pipe.check_status()
    assert pipe.prefill_launches == 6
    o, st, dense = pipe.o.clone(), pipe.plan_st.info.n_units, pipe.plan_dense.info.n_units
    pipe.build_plans()
    assert (st, dense) == (pipe.plan_st.info.n_units, pipe.plan_dense.info.n_units) and pipe.plan_st.info.max_chunks > 1
    for n in range(6):
        pipe.prefill_layer(n, q[n], k[n], v[n])
    assert torch.equal(pipe.o, o)
