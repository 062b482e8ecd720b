"""The work this library is measured on: whole passes over a prompt, and its steps one at a time.

A case is a dict of plain values.  `kind` names the call:

    pass      a prompt from Q/K/V to its first decoded token: plans, every layer's prefill, the window scores, selection
              and compaction (PureKVPipeline.run_device), then one decode step over each compacted layer's cache
    prefill   one layer's attention with its plan in hand
    score     one layer's key scores: `form` lse (one pass, from the dense prefill's log-sum-exp), window (two passes,
              computes it itself) or observe (the last 32 rows vote, pooled over 7 keys)
    compress  V-norm weighting, top-h selection and compaction of many layers from one layer's scores
    decode    one decode step over the compact caches of `layers` layers, one call per layer

A batch is `n_req` requests of `prefix` text tokens, a number of frames of grid_h x grid_w visual tokens and some more
text, the last two drawn per request between the given limits with `shape_seed`.

Q/K/V are N(0, 1); 5 % of the visual keys and the last 16 queries of each request share a direction (`inputs.py` holds the
same recipe for the parity tests), so the scores have the few heavy keys that selection is about.
"""
import math
import random

import torch

from paper_2510_25600_b200 import binding as P
from paper_2510_25600_b200 import inputs
from paper_2510_25600_b200.pipeline import PureKVPipeline

OBS_ROWS, POOL = 32, 7   # the observation window and its pooling, as the reduction benchmarks of bench.py set them
LOCAL_WINDOW = 256       # the local mask's window, likewise

VIDEOLLAMA2 = dict(heads=32, kv_heads=8, head_dim=128, dtype="bf16", grid_h=12, grid_w=12, tile=64, window=64)
QWEN25VL = dict(heads=28, kv_heads=4, head_dim=128, dtype="bf16", grid_h=16, grid_w=16, tile=128, window=64)


def _batch(n_req, prefix, frames, text, shape_seed=0):
    return dict(n_req=n_req, prefix=prefix, frames_lo=frames[0], frames_hi=frames[1], text_lo=text[0], text_hi=text[1],
                shape_seed=shape_seed)


def listed():
    ragged = dict(QWEN25VL, window=32, **_batch(8, 0, (8, 64), (32, 256), 4))
    long_video = dict(QWEN25VL, grid_h=24, grid_w=24, window=256, **_batch(1, 0, (64, 64), (256, 256)))
    return [
        # The smallest prompt: a short clip in fp32 on the CUDA-core path, where launches and host work are everything.
        dict(name="tiny_fp32_pass", kind="pass", heads=2, kv_heads=1, head_dim=64, dtype="fp32", grid_h=8, grid_w=8, tile=16,
             window=16, keep=0.2, layers=1, scored=1, dense_layers=0, **_batch(1, 16, (4, 4), (16, 16))),
        # An ordinary prompt of a 32-layer model: 16 frames, 2432 tokens; layer 0 scores, 31 layers are compacted.
        dict(VIDEOLLAMA2, name="videollama2_pass", kind="pass", keep=0.2, layers=32, scored=1, dense_layers=1,
             **_batch(1, 64, (16, 16), (64, 64))),
        # The headline prompt: 32 frames, 8320 tokens, 28 layers; layers 0-1 score, 26 layers are compacted.
        dict(QWEN25VL, name="qwen25vl_pass", kind="pass", keep=0.2, layers=28, scored=2, dense_layers=2,
             **_batch(1, 64, (32, 32), (64, 64))),
        # One sparse layer of a long video: 64 frames of 24 x 24, 37 120 tokens.
        dict(long_video, name="long_video_prefill", kind="prefill", mask="st"),
        # One sparse layer of a ragged serving batch: 8 requests of 8-64 frames.
        dict(ragged, name="ragged_prefill", kind="prefill", mask="st"),
        # The scored layer of that batch: dense causal attention that also leaves the rows' log-sum-exp.
        dict(ragged, name="ragged_prefill_dense", kind="prefill", mask="dense"),
        # Key scores of the long video from the dense prefill's log-sum-exp, with its wide recent window.
        dict(long_video, name="long_video_score", kind="score", form="lse"),
        # Key scores without a log-sum-exp at hand, the reduction of observation-window policies, an ordinary prompt.
        dict(VIDEOLLAMA2, name="observed_score", kind="score", form="observe", **_batch(1, 64, (16, 16), (64, 64))),
        # Compression of the headline prompt's 26 layers: few long segments.
        dict(QWEN25VL, name="qwen25vl_compress", kind="compress", keep=0.2, layers=26, **_batch(1, 64, (32, 32), (64, 64))),
        # Compression of the ragged batch's 27 layers: many segments of uneven length.
        dict(ragged, name="ragged_compress", kind="compress", keep=0.2, layers=27),
        # A decoded token of one conversation: 26 layers' compact caches of 1664 rows, where latency counts.
        dict(QWEN25VL, name="decode_one", kind="decode", keep=0.2, layers=26, **_batch(1, 64, (32, 32), (64, 64))),
        # A decoded token of 128 conversations at once, one layer: 2900-5100 kept rows each, where bandwidth counts.
        dict(QWEN25VL, name="decode_batch", kind="decode", keep=0.2, layers=1, **_batch(128, 64, (56, 100), (32, 256), 7)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pass", "pass", "prefill", "prefill", "score", "compress", "decode"])
    if kind == "pass" and rng.random() < 0.25:  # the fp32 path: short prompts
        gh, gw = rng.randint(5, 9), rng.randint(5, 9)
        return dict(kind="pass", heads=2, kv_heads=1, head_dim=64, dtype="fp32", grid_h=gh, grid_w=gw, tile=rng.choice([16, 32]),
                    window=rng.choice([8, 11, 16]), keep=rng.choice([0.1, 0.2, 0.5]), layers=rng.randint(1, 3), scored=1,
                    dense_layers=0, **_batch(1, rng.randint(0, 24), (2, rng.randint(2, 6)), (16, rng.randint(17, 48)),
                                             rng.randrange(1000)))
    c = dict(rng.choice([VIDEOLLAMA2, QWEN25VL]), kind=kind)
    side = rng.randint(8, 24)
    c.update(grid_h=side, grid_w=rng.randint(max(6, side - 4), side + 3), tile=rng.choice([64, 128]))
    n = c["grid_h"] * c["grid_w"]
    # tokens in all, over the range of the listed batches of that kind
    lo, hi = {"pass": (600, 8000), "prefill": (600, 36000), "score": (600, 36000), "compress": (600, 60000),
              "decode": (600, 1000000)}[kind]
    tokens = _log_int(rng, lo, hi)
    n_req = 1 if rng.random() < 0.4 else _log_int(rng, 2, 128 if kind == "decode" else 8)
    n_req = min(n_req, max(1, tokens // (2 * n)))
    mean = max(1, tokens // (n_req * n))
    spread = 0 if n_req == 1 else rng.randint(0, mean // 2)
    text = rng.randint(20, 160)
    c.update(_batch(n_req, rng.choice([0, 0, rng.randint(1, 90)]), (max(1, mean - spread), mean + spread), (text, text + rng.randint(0, 120)),
                    rng.randrange(1000)))
    # a window that is a multiple of 8 takes the one-pass scores, any other the two passes
    c["window"] = rng.choice([16, 32, 64, 64, 128, rng.randint(9, 100)])
    c["keep"] = rng.choice([0.05, 0.1, 0.2, 0.2, 0.35, 0.5])
    if kind == "pass":
        c.update(scored=rng.randint(1, 2), layers=min(rng.randint(3, 28), max(3, 28 * 6000 // tokens)))
        c["dense_layers"] = c["scored"]
    elif kind == "prefill":
        c["mask"] = rng.choice(["st", "st", "spatial", "local"] + (["dense"] if tokens < 12000 else []))
    elif kind == "score":
        c["form"] = rng.choice(["lse", "lse", "window", "observe"])
        if c["form"] == "lse":
            c["window"] = min(c["window"], c["frames_lo"] * n + text) // 8 * 8
    elif kind == "compress":
        c["layers"] = max(2, min(rng.randint(4, 31), 27 * 60000 // tokens))
    else:
        c["layers"] = max(1, min(rng.randint(1, 31), 500000 // tokens))
    return c


# ---- the shapes a case stands for --------------------------------------------------------------------------------------
def _shape(case):
    rng = random.Random(case["shape_seed"])
    n = case["grid_h"] * case["grid_w"]
    frames = [rng.randint(case["frames_lo"], case["frames_hi"]) for _ in range(case["n_req"])]
    text = [rng.randint(case["text_lo"], case["text_hi"]) for _ in range(case["n_req"])]
    prefix = [case["prefix"]] * case["n_req"]
    lens = [case["prefix"] + f * n + t for f, t in zip(frames, text)]
    return lens, prefix, frames


def _mask(case, name):
    if name == "dense":
        return inputs.STMask(case["grid_h"], case["grid_w"], tile=case["tile"], dense_causal=True)
    return inputs.mask_variant(name, case["grid_h"], case["grid_w"], tile=case["tile"], local_window=LOCAL_WINDOW)


def _pairs(case, name):
    """(query, key) pairs the mask keeps, all requests of the batch."""
    n, total = case["grid_h"] * case["grid_w"], 0
    causal = lambda first, last: (last * (last + 1) - first * (first + 1)) // 2  # positions first .. last - 1 see i + 1 keys
    for length, pre, frames in zip(*_shape(case)):
        end = pre + frames * n
        if name == "dense":
            total += causal(0, length)
            continue
        total += causal(0, pre) + causal(end, length)
        if name == "local":
            v = frames * n
            total += v * pre + causal(0, min(v, LOCAL_WINDOW)) + max(0, v - LOCAL_WINDOW) * LOCAL_WINDOW
            continue
        for f in range(frames):  # prefix, first frame, own frame up to the diagonal, the cell of the previous frame
            total += n * pre + causal(0, n)
            total += n * n if f >= 1 else 0
            total += n if f >= 2 and name == "st" else 0
    return total


def _kept(case, lens):
    return [P.purekv_budget(length, case["window"], case["keep"])[1] for length in lens]


def work(case):
    lens, _, _ = _shape(case)
    t, h, hkv, d = sum(lens), case["heads"], case["kv_heads"], case["head_dim"]
    esz = 2 if case["dtype"] == "bf16" else 4
    q_row, kv_row = h * d * esz, 2 * hkv * d * esz  # bytes of a token's Q (or O), and of its K and V, in one layer
    kind, layers = case["kind"], case.get("layers", 1)
    if kind == "prefill":
        return {"bytes": t * (2 * q_row + kv_row) + (4 * h * t if case["mask"] == "dense" else 0),
                "flops": 4.0 * d * h * _pairs(case, case["mask"])}
    if kind == "score":
        rows = OBS_ROWS if case["form"] == "observe" else case["window"]
        voting = sum(min(rows, length) for length in lens)
        return {"bytes": t * kv_row // 2 + voting * q_row + 4 * hkv * t + (4 * h * voting if case["form"] == "lse" else 0),
                "flops": (2.0 if case["form"] == "lse" else 4.0) * h * d * sum(min(rows, length) * length for length in lens)}
    kept = _kept(case, lens)
    if kind == "compress":  # scores and V once, the indices, and the kept rows read (K; V is at hand) and written
        return {"bytes": 4 * hkv * t + layers * (t * kv_row // 2 + sum(kept) * (4 * hkv + kv_row // 2 + kv_row)),
                "flops": 2.0 * layers * t * hkv * d}
    if kind == "decode":
        return {"bytes": layers * (sum(kept) * kv_row + 2 * len(lens) * q_row), "flops": 4.0 * layers * d * h * sum(kept)}
    dense, compacted = case["dense_layers"], layers - case["dense_layers"]
    return {"bytes": layers * t * (2 * q_row + kv_row) + compacted * (sum(kept) * kv_row + 2 * len(lens) * q_row) + 4 * hkv * t * case["scored"],
            "flops": 4.0 * d * h * (max(dense, 1) * _pairs(case, "dense") + (layers - max(dense, 1)) * _pairs(case, "st")) +
            case["scored"] * 2.0 * h * d * sum(min(case["window"], length) * length for length in lens) + compacted * 4.0 * d * h * sum(kept)}


def tolerance(case):
    kind = case["kind"]
    if kind == "compress":
        return "exact"  # whole positions and copied rows
    # about four times what each path shows against the same computation in 64 bits (rel / max in brackets)
    if case["dtype"] == "fp32":
        return {"rel": 1e-6, "max": 1e-5}  # [2.6e-7 / 2e-6]
    if kind == "score":
        # exact products, 32-bit sums, and a share of exponentials that may be a cubic [2.3e-6 / 1e-5]
        return {"rel": 1e-5, "max": 4e-5}
    if kind == "decode":
        return {"rel": 8e-3, "max": 0.04}  # bf16 weights and outputs [2.3e-3 / 9e-3]
    if kind == "prefill":
        return {"rel": 1e-2, "max": 0.25}  # bf16 probabilities and outputs [2.3e-3 / 6e-2]
    # As prefill; and where a score moves by its last bits a key at the selection's threshold may change places with its
    # neighbour, which the decoded token shows as one key of some hundreds exchanged.
    return {"rel": 1e-2, "max": 0.5}


# ---- inputs ------------------------------------------------------------------------------------------------------------
def _marks(case, gen):
    """Which tokens are salient keys, and which are among the last 16 queries of their request."""
    lens, prefix, frames = _shape(case)
    n = case["grid_h"] * case["grid_w"]
    visual = torch.zeros(sum(lens), dtype=torch.bool)
    last = torch.zeros_like(visual)
    at = 0
    for length, pre, f in zip(lens, prefix, frames):
        visual[at + pre:at + pre + f * n] = True
        last[max(at, at + length - 16):at + length] = True
        at += length
    salient = visual.cuda() & (torch.rand(visual.numel(), generator=gen, device="cuda") < 0.05)
    return salient, last.cuda()


def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)


def _qkv(case, gen, layers, which="qkv"):
    """Q [layers, T, H, d], K and V [layers, T, H_kv, d]; only those named are made."""
    t, h, hkv, d = sum(_shape(case)[0]), case["heads"], case["kv_heads"], case["head_dim"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    salient, last = _marks(case, gen)
    out = {name: torch.empty((layers, t, h if name == "q" else hkv, d), dtype=dt, device="cuda") for name in which}
    for layer in range(layers):
        u = _normal(gen, hkv, d)
        u = u / u.norm(dim=1, keepdim=True)
        for name in which:
            x = _normal(gen, t, h if name == "q" else hkv, d)
            if name == "k":
                x += salient[:, None, None] * 3.0 * u
            elif name == "q":
                x += last[:, None, None] * u.repeat_interleave(h // hkv, dim=0)
            out[name][layer] = x
    return [out[name] for name in which]


def _row_lse(case, q, k):
    """Log-sum-exp of the window rows' causal logits, as the dense prefill leaves it (other rows are not read)."""
    h, g = case["heads"], case["heads"] // case["kv_heads"]
    lse = torch.zeros((h, q.shape[0]), dtype=torch.float32, device="cuda")
    at = 0
    for length in _shape(case)[0]:
        w = min(case["window"], length)
        rows = torch.arange(length - w, length, device="cuda")
        hidden = torch.arange(length, device="cuda")[None, :] > rows[:, None]
        for head in range(h):
            s = q[at + length - w:at + length, head].float() @ k[at:at + length, head // g].float().T / math.sqrt(case["head_dim"])
            lse[head, at + length - w:at + length] = torch.logsumexp(s.masked_fill_(hidden, -math.inf), dim=1)
        at += length
    return lse


def _scores(case, gen):
    """Positive key scores as Eq. 1-2 give them: a log-normal body and a few salient keys well above it."""
    lens = _shape(case)[0]
    salient, _ = _marks(case, gen)
    c = torch.exp(0.3 * _normal(gen, case["kv_heads"], sum(lens))) * (1.0 + 2.0 * salient)
    at = 0
    for length in lens:
        w = min(case["window"], length)
        c[:, at:at + length] *= w / length
        c[:, at + length - w:at + length] = 0.0
        at += length
    return c


def _decode_ws(case, lens):
    need = P.purekv_decode_ws_bytes(len(lens), max(_kept(case, lens)), case["heads"], case["kv_heads"], case["head_dim"])
    return torch.empty(max(16, need), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    lens, prefix, frames = _shape(case)
    kind, h, hkv, d = case["kind"], case["heads"], case["kv_heads"], case["head_dim"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    s = dict(case=case)
    if kind == "pass":
        layers, first = case["layers"], case["dense_layers"]
        s["pipe"] = PureKVPipeline(lens, prefix, frames, _mask(case, "st"), layers, h, hkv, d, dt, tuple(range(case["scored"])),
                                   tuple(range(first, layers)), case["window"], case["keep"])
        s["q"], s["k"], s["v"] = _qkv(case, gen, layers)
        s["q_next"] = 1.5 * _normal(gen, layers - first, len(lens), h, d)
        s["q_next"] = s["q_next"].to(dt)
        s["o_next"] = torch.empty_like(s["q_next"])
        s["ws"] = _decode_ws(case, lens)
        return s
    s["batch"] = batch = P.Batch(lens, prefix, frames)
    s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    if kind == "prefill":
        s["q"], s["k"], s["v"] = (x[0] for x in _qkv(case, gen, 1))
        s["plan"] = P.purekv_plan_build(batch, P.st_params(_mask(case, case["mask"])), P.BF16, d, h, hkv)
        s["o"] = torch.empty_like(s["q"])
        s["lse"] = torch.empty((h, sum(lens)), dtype=torch.float32, device="cuda") if case["mask"] == "dense" else None
        s["ws"] = torch.empty(max(16, s["plan"].info.ws_bytes), dtype=torch.uint8, device="cuda")
        return s
    if kind == "score":
        s["q"], s["k"] = (x[0] for x in _qkv(case, gen, 1, "qk"))
        s["c"] = torch.empty((hkv, sum(lens)), dtype=torch.float32, device="cuda")
        if case["form"] == "lse":
            s["lse"] = _row_lse(case, s["q"], s["k"])
        else:
            need = (P.purekv_score_ws_bytes(batch, case["window"], h) if case["form"] == "window" else
                    P.purekv_score_ex_ws_bytes(batch, OBS_ROWS, POOL, h, hkv))
            s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
        return s
    s["budget"] = budget = P.Budget(batch, case["window"], case["keep"])
    layers = case["layers"]
    if kind == "compress":
        s["c"] = _scores(case, gen)
        s["k"], s["v"] = _qkv(case, gen, layers, "kv")
        s["idx"] = torch.empty((layers, hkv, budget.total_kept), dtype=torch.int32, device="cuda")
        s["k_c"] = torch.empty((layers, budget.total_kept, hkv, d), dtype=dt, device="cuda")
        s["v_c"] = torch.empty_like(s["k_c"])
        s["ws"] = torch.empty(P.purekv_select_ws_bytes(batch, layers, hkv), dtype=torch.uint8, device="cuda")
        return s
    cache = lambda: torch.stack([_normal(gen, budget.total_kept, hkv, d).to(dt) for _ in range(layers)])
    s["k_c"], s["v_c"] = cache(), cache()
    s["q"] = (1.5 * _normal(gen, layers, len(lens), h, d)).to(dt)
    s["o"] = torch.empty_like(s["q"])
    s["ws"] = _decode_ws(case, lens)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "pass":
        pipe = s["pipe"]
        pipe.run_device(s["q"], s["k"], s["v"])
        for n in range(len(pipe.compacted)):
            P.purekv_decode_attention(s["q_next"][n], pipe.k_c[n], pipe.v_c[n], pipe.budget, out=s["o_next"][n], ws=s["ws"])
        return {"o": pipe.o, "c": pipe.c, "o_next": s["o_next"]}
    if kind == "prefill":
        P.purekv_st_sparse_prefill(s["q"], s["k"], s["v"], s["batch"], s["plan"], out=s["o"], lse=s["lse"], status=s["status"],
                                   ws=s["ws"])
        return {"o": s["o"], "lse": s["lse"]}
    if kind == "score":
        if case["form"] == "lse":
            return P.purekv_lowlayer_score_lse(s["q"], s["k"], s["lse"], s["batch"], case["window"], c_out=s["c"], status=s["status"])
        if case["form"] == "window":
            return P.purekv_lowlayer_score(s["q"], s["k"], s["batch"], case["window"], c_out=s["c"], ws=s["ws"])
        return P.purekv_lowlayer_score_ex(s["q"], s["k"], s["batch"], case["window"], OBS_ROWS, POOL, c_out=s["c"], ws=s["ws"])
    if kind == "compress":
        P.purekv_select_topk(s["c"], s["v"], s["batch"], s["budget"], idx_out=s["idx"], ws=s["ws"])
        P.purekv_compact_kv(s["k"], s["v"], s["idx"], s["batch"], s["budget"], k_out=s["k_c"], v_out=s["v_c"])
        return {"idx": s["idx"], "k": s["k_c"], "v": s["v_c"]}
    for layer in range(case["layers"]):
        P.purekv_decode_attention(s["q"][layer], s["k_c"][layer], s["v_c"][layer], s["budget"], out=s["o"][layer], ws=s["ws"])
    return s["o"]
