"""One pass of the PureKV hot path over a batch: the sequence of C-ABI calls a caller makes.

    layers <= CLIE layer : dense causal prefill; the CLIE layer also yields the window scores C
    higher layers        : ST-SpAttn prefill
    then                 : V-norm weighting + top-h selection and K/V compaction of the
                           compressed layers

This module only sequences calls of `binding` and owns the device buffers (torch); it does
no arithmetic of the method.  `run_host` is the end-to-end form: inputs start in pinned host
memory and the compact cache is read back to the host.
"""
from __future__ import annotations

from typing import Optional, Sequence

import torch

from . import binding as P


class PureKVPipeline:
    def __init__(self, seq_lens: Sequence[int], n_prefix: Sequence[int], n_frames: Sequence[int], mask,
                 n_layers: int, n_q_heads: int, n_kv_heads: int, head_dim: int, dtype: torch.dtype,
                 scored_layers: Sequence[int], compacted_layers: Sequence[int], window: int, keep_ratio: float,
                 kv_layers: Optional[int] = None):
        """`mask` has the STMask attributes.  Layers up to max(scored_layers) run dense causal attention,
        the rest ST-SpAttn.  K/V exist for kv_layers >= n_layers layers (default n_layers)."""
        self.mask, self.n_layers = mask, n_layers
        self.h, self.hkv, self.d, self.dtype = n_q_heads, n_kv_heads, head_dim, dtype
        self.code = P.BF16 if dtype == torch.bfloat16 else P.FP32
        self.clie = max(scored_layers)
        self.scored = tuple(scored_layers)
        self.compacted = tuple(compacted_layers)
        assert self.compacted == tuple(range(self.compacted[0], self.compacted[-1] + 1)), "compacted layers must be contiguous"
        self.kv_layers = kv_layers if kv_layers is not None else max(n_layers, self.compacted[-1] + 1)
        self.window, self.keep_ratio = window, keep_ratio
        self.batch = P.Batch(seq_lens, n_prefix, n_frames)
        self.budget = P.Budget(self.batch, window, keep_ratio)
        t = self.batch.total_tokens
        dev = "cuda"
        params_dense = P.st_params(mask)
        params_dense.flags |= P.FLAG_DENSE_CAUSAL
        self.params_dense, self.params_st = params_dense, P.st_params(mask)
        hh = (n_q_heads, n_kv_heads)
        self.n_dense = min(n_layers, self.clie + 1)
        self.n_sparse = n_layers - self.n_dense
        # room for a plan of all layers under the mask (run_device) and for one of a layer at a time (build_plans, prefill_layer)
        plan_buf = lambda params, layers: torch.empty(
            max(1, P.purekv_plan_bytes(self.batch, params, self.code, head_dim, *hh, n_layers=max(1, layers))), dtype=torch.uint8,
            device=dev)
        self.plan_buf_dense, self.plan_buf_st = plan_buf(params_dense, self.n_dense), plan_buf(self.params_st, self.n_sparse)
        self.prefill_ws = None
        # per mask a ring of pinned buffers, each with the event behind its last copy; the last one used comes first
        self._h_dense, self._h_st = ([[torch.empty(b.numel(), dtype=torch.uint8, pin_memory=True), None] for _ in range(3)]
                                     for b in (self.plan_buf_dense, self.plan_buf_st))
        self._copies = torch.cuda.Stream()  # the sparse plan's copy runs beside the dense layers
        self.o = torch.empty((n_layers, t, n_q_heads, head_dim), dtype=dtype, device=dev)
        self.c = torch.empty((len(self.scored), n_kv_heads, t), dtype=torch.float32, device=dev)
        # one-pass tensor-core scores where the entry point supports the shape (bf16, head_dim 128, window and any
        # clipped window a multiple of 8); the two-pass kernels otherwise
        self.one_pass_scores = (dtype == torch.bfloat16 and head_dim == 128 and window % 8 == 0 and
                                all(l >= window or l % 8 == 0 for l in seq_lens))
        # rows' log-sum-exp, a layer after the other: of every dense layer, so that one call takes them all, scored or not
        self._lse = torch.empty((self.n_dense if self.one_pass_scores else 0, n_q_heads, t), dtype=torch.float32, device=dev)
        self.score_ws = torch.empty(P.purekv_score_ws_bytes(self.batch, window, n_q_heads), dtype=torch.uint8, device=dev)
        nc = len(self.compacted)
        self.select_ws = torch.empty(P.purekv_select_ws_bytes(self.batch, nc, n_kv_heads), dtype=torch.uint8, device=dev)
        self.idx = torch.empty((nc, n_kv_heads, self.budget.total_kept), dtype=torch.int32, device=dev)
        self.k_c = torch.empty((nc, self.budget.total_kept, n_kv_heads, head_dim), dtype=dtype, device=dev)
        self.v_c = torch.empty_like(self.k_c)
        self.status = torch.zeros(1, dtype=torch.int32, device=dev)
        self.plan_dense = self._plan_st = None
        self.prefill_launches = n_layers  # of the last pass (before the first: a layer at a time)

    @property
    def launches_per_step(self) -> int:
        """Kernels of the last pass: prefill, score (1 one-pass or in one cluster, up to 3 otherwise: counted as 1), select (2),
        compact."""
        return self.prefill_launches + len(self.scored) + 2 + 1

    @property
    def lse(self) -> torch.Tensor:
        """[scored layers, H, T]: the log-sum-exp that the one-pass scores read."""
        first, last = self.scored[0], self.scored[-1]
        return self._lse[first:last + 1] if self.scored == tuple(range(first, last + 1)) else self._lse[list(self.scored)]

    def _plan(self, params, ring: list, d_buf: torch.Tensor, layers: int = 1) -> P.Plan:
        """Plans one mask, for launches of `layers` layers, on the host into a pinned buffer and enqueues its copy on the
        current stream without waiting, so planning overlaps the GPU work already in flight.  A small ring of pinned buffers
        keeps a plan alive until its copy has run."""
        ring.append(ring.pop(0))
        h_buf, ev = ring[0]
        if ev is not None:
            ev.synchronize()
        else:
            ev = ring[0][1] = torch.cuda.Event()
        _, info = P.purekv_plan_build_host(self.batch, params, self.code, self.d, self.h, self.hkv, out=h_buf,
                                           n_layers=layers)
        d_buf.copy_(h_buf, non_blocking=True)
        ev.record()
        return P.Plan(d_buf, info)

    @property
    def plan_st(self) -> P.Plan:
        """The sparse mask's plan.  A pass without sparse layers does not need it: it is then made when asked for."""
        if self._plan_st is None:
            self._plan_st = self._plan(self.params_st, self._h_st, self.plan_buf_st)
            self._size_prefill_ws(self._plan_st)
        return self._plan_st

    def _size_prefill_ws(self, plan: P.Plan) -> None:
        need = max(16, plan.info.ws_bytes)
        if self.prefill_ws is None or self.prefill_ws.numel() < need:
            self.prefill_ws = torch.empty(need, dtype=torch.uint8, device="cuda")

    def build_plans(self) -> None:
        """Both masks' plans, for `prefill_layer` calls; `run_device` builds its own, each just ahead of the first layer that
        needs it."""
        self.plan_dense = self._plan(self.params_dense, self._h_dense, self.plan_buf_dense)
        self._plan_st = self._plan(self.params_st, self._h_st, self.plan_buf_st)
        self._size_prefill_ws(self.plan_dense)
        self._size_prefill_ws(self.plan_st)

    def prefill_layer(self, layer: int, q: torch.Tensor, k: torch.Tensor, v: torch.Tensor) -> None:
        plan = self.plan_dense if layer <= self.clie else self.plan_st
        # a scored layer is dense causal: its prefill also leaves the rows' log-sum-exp for the one-pass scores
        lse = self._lse[layer] if (self.one_pass_scores and layer in self.scored) else None
        P.purekv_st_sparse_prefill(q, k, v, self.batch, plan, out=self.o[layer], lse=lse, status=self.status,
                                   ws=self.prefill_ws)

    def _share_launches(self, q, k, v) -> bool:
        """Whether Q/K/V are stacked layers that one launch can take (a sequence of layers has no stacked views, and layers that
        overlap, one for all of them, say, are launches of their own)."""
        t = self.batch.total_tokens
        return (isinstance(q, torch.Tensor) and isinstance(k, torch.Tensor) and isinstance(v, torch.Tensor) and
                q.stride(0) >= t * self.h * self.d and k.stride(0) == v.stride(0) >= t * self.hkv * self.d)

    def _prefill(self, plan: P.Plan, lo: int, hi: int, q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, shared: bool, events) -> None:
        """Layers lo .. hi - 1, all under one mask: in one call (`shared`), which is one launch if the plan is the tensor-core
        kernel's and leaves lists whole, or one by one, each between its pair of `events` if those are given."""
        if shared:
            lse = self._lse[lo:hi] if self.one_pass_scores and lo < self.n_dense else None
            P.purekv_st_sparse_prefill_layers(q[lo:hi], k[lo:hi], v[lo:hi], self.batch, plan, out=self.o[lo:hi], lse=lse,
                                              status=self.status, ws=self.prefill_ws)
            self.prefill_launches += 1 if plan.info.n_units > 0 and plan.info.max_chunks == 1 else hi - lo
            return
        for layer in range(lo, hi):
            if events is not None:
                events[layer][0].record()
            self.prefill_layer(layer, q[layer], k[layer], v[layer])
            if events is not None:
                events[layer][1].record()
        self.prefill_launches += hi - lo

    def run_device(self, q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, events=None, marks=None) -> None:
        """q [n_layers,T,H,d], k,v [kv_layers,T,H_kv,d] on the GPU.  Results in self.o / idx / k_c / v_c.
        `events`, if given, is a list of (start, end) torch.cuda.Event pairs, one per layer, which is then a prefill launch
        of its own, as it is where Q is a sequence of layers; the layers of a stacked Q are one launch per mask where the plan
        allows it.  `marks`, if given, is three events recorded before the first prefill launch, after the last dense-causal one and after the last one."""
        # The sparse mask's plan, the longer one, is made and copied while the GPU works on the dense layers.  (The copy
        # waits for whatever the stream held before this call, which may still read the last plan; in the stream itself,
        # between two layers, it cost 10 us.)
        before = torch.cuda.Event() if self.n_sparse else None
        if before is not None:
            before.record()
        # planned for the launches that are made: lists that are left whole for one launch end unevenly in a launch per layer
        shared = events is None and (self.n_dense > 1 or self.n_sparse > 1) and self._share_launches(q, k, v)
        self.prefill_launches = 0
        self.plan_dense = self._plan(self.params_dense, self._h_dense, self.plan_buf_dense, self.n_dense if shared else 1)
        self._size_prefill_ws(self.plan_dense)
        if marks is not None:
            marks[0].record()
        self._prefill(self.plan_dense, 0, self.n_dense, q, k, v, shared and self.n_dense > 1, events)
        if marks is not None:
            marks[1].record()
        if before is not None:
            main = torch.cuda.current_stream()
            self._copies.wait_event(before)
            with torch.cuda.stream(self._copies):
                self._plan_st = self._plan(self.params_st, self._h_st, self.plan_buf_st, self.n_sparse if shared else 1)
            main.wait_event(self._h_st[0][1])
            self._size_prefill_ws(self._plan_st)
            self._prefill(self._plan_st, self.n_dense, self.n_layers, q, k, v, shared and self.n_sparse > 1, events)
        if marks is not None:
            marks[2].record()
        for n, layer in enumerate(self.scored):
            if self.one_pass_scores:
                P.purekv_lowlayer_score_lse(q[layer], k[layer], self._lse[layer], self.batch, self.window, c_out=self.c[n],
                                            status=self.status)
            else:
                P.purekv_lowlayer_score(q[layer], k[layer], self.batch, self.window, c_out=self.c[n], ws=self.score_ws)
        lo, hi = self.compacted[0], self.compacted[-1] + 1
        k_cmp, v_cmp = k[lo:hi], v[lo:hi]
        P.purekv_select_topk(self.c[len(self.scored) - 1], v_cmp, self.batch, self.budget, idx_out=self.idx,
                             ws=self.select_ws)
        P.purekv_compact_kv(k_cmp, v_cmp, self.idx, self.batch, self.budget, k_out=self.k_c, v_out=self.v_c)

    def alloc_host_io(self):
        """Pinned host buffers for run_host: (q, k, v) inputs and (k_c, v_c, o_last) outputs."""
        t = self.batch.total_tokens
        pin = dict(dtype=self.dtype, pin_memory=True)
        ins = (torch.empty((self.n_layers, t, self.h, self.d), **pin),
               torch.empty((self.kv_layers, t, self.hkv, self.d), **pin),
               torch.empty((self.kv_layers, t, self.hkv, self.d), **pin))
        outs = (torch.empty(tuple(self.k_c.shape), **pin), torch.empty(tuple(self.v_c.shape), **pin),
                torch.empty((t, self.h, self.d), **pin))
        return ins, outs

    def run_host(self, h_in, h_out, d_in) -> None:
        """End to end: pinned host Q/K/V -> device (d_in, caller-owned staging) -> hot path -> compact cache and
        the last layer's O back in pinned host memory.  Synchronises before returning."""
        for src, dst in zip(h_in, d_in):
            dst.copy_(src, non_blocking=True)
        self.run_device(*d_in)
        h_out[0].copy_(self.k_c, non_blocking=True)
        h_out[1].copy_(self.v_c, non_blocking=True)
        h_out[2].copy_(self.o[self.n_layers - 1], non_blocking=True)
        torch.cuda.current_stream().synchronize()

    def check_status(self) -> None:
        P.purekv_poll_status(self.status)
