"""The work whose speed this repository is measured on, case by case.

Every case goes through the entry points of the ctypes binding (paper_2609_37007_gb300.mcd):

  frames    one audio frame c1..c15 of one stream or of many (mcd_decode_frame,
            mcd_decode_frame_host, mcd_decode_frames), chain drafts or a sparse tree, bf16, W8A16
            or fp32 weights;
  prefill   a text prompt through the 28-layer CodeDecoder (mcd_outer_prefill);
  rows      the CodeDecoder's rows of the frames that follow (mcd_outer_step);
  gemm      an activation matrix laid out and multiplied by laid-out weights on the tensor
            cores (mcd_tc_tile, mcd_tc_gemm_tiled);
  topk      top-k / temperature distributions of logits rows (mcd_topk_softmax_static).

The model's shapes and sampling are those of `synth` (MCD, TINY, OUTER).  Its weights are
drawn here once per process and kept with their context, as a program that serves a model
keeps them; the inputs of a pass come from the seed.  The weights are random with one thing
that trained weights have and random ones lack: confident predictions.  Code c at position
s - 1 predicts code (c + 37 s) mod V at position s: LM head s has that code's embedding row
added to the predicted row, and the same for the positions the drafts look ahead from, so the
top logit stands clear of the others and a draft is right or wrong for a reason (the first
draft always, later ones for even codes only: 2.75 tokens per call at K = 3).  What a frame
emits then does not hang on the last bits of a sum, so two correct implementations feed the same
rows, call by call, and their logits can be compared to the end of the frame.
"""
import math

import numpy as np
import torch

from paper_2609_37007_gb300 import mcd, synth

SHIFT = 37            # code c at position s - 1 predicts (c + SHIFT s) mod V at position s
WRONG = 999           # a wrong draft proposes the code this far past the right one
SIBLING = 411         # the rank-r candidate of a tree's drafts is r * SIBLING past the right code
PEAK = 32.0           # logit of a predicted code
RANKS = (1.0, 0.55, 0.5, 0.45)   # strength of a tree's candidates by rank
TREE_DEPTH = 3


# ---- the cases ---------------------------------------------------------------------------
def listed():
    frame = dict(kind="frame", streams=1, slots=1, draft_len=3, dtype="bf16", model="mcd", nodes=0, host=False)
    return [
        # the distributions of one batched call's rows: the smallest call, all latency
        dict(name="topk_128x2048", kind="topk", rows=128, vocab=2048, top_k=50),
        # the gate/up product of 128 streams x 4 rows
        dict(name="gemm_6144x512x1024", kind="gemm", m=6144, n=512, k=1024),
        # the small fp32 model: weights in L2, so launches and hand-offs are all there is
        dict(frame, name="frame_tiny_f32", model="tiny", dtype="f32", draft_len=2),
        # one interactive stream with the position-aware drafter: the workload of bench.py
        dict(frame, name="frame_k3"),
        # plain autoregressive decoding from host buffers: a host-driven TTS loop
        dict(frame, name="frame_ar_host", draft_len=0, host=True),
        # 8-bit weights with a longer draft
        dict(frame, name="frame_int8_k5", draft_len=5, dtype="int8"),
        # the sparse tree of the paper's headline: 32 nodes, 33 rows per call
        dict(frame, name="frame_tree32", nodes=32),
        # a few streams sharing the weights
        dict(frame, name="streams_3", streams=3, slots=4),
        dict(frame, name="streams_8", streams=8, slots=8),
        # a server's full batch: 512 packed rows per call
        dict(frame, name="streams_128", streams=128, slots=128),
        # a 256-token prompt before the first frame
        dict(name="prefill_256", kind="prefill", tokens=256),
        # the CodeDecoder's rows of 12 frames over a cache of a few hundred positions
        dict(name="rows_12_at_333", kind="rows", tokens=333, rows=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["topk", "gemm", "frame", "frame", "tree", "streams", "streams", "prefill", "rows"])
    if kind == "topk":
        vocab = 16 * _log_int(rng, 4, 256)
        return dict(kind="topk", rows=_log_int(rng, 1, 128), vocab=vocab, top_k=min(vocab, _log_int(rng, 1, 128)))
    if kind == "gemm":
        return dict(kind="gemm", m=128 * _log_int(rng, 1, 64), n=16 * _log_int(rng, 1, 64), k=64 * _log_int(rng, 1, 48))
    if kind == "prefill":
        return dict(kind="prefill", tokens=_log_int(rng, 2, 480))
    if kind == "rows":
        return dict(kind="rows", tokens=_log_int(rng, 1, 480), rows=rng.randint(2, 10))
    case = dict(kind="frame", streams=1, slots=1, draft_len=3, dtype="bf16", model="mcd", nodes=0, host=False)
    if kind == "tree":
        case.update(nodes=_log_int(rng, 4, 64))
    elif kind == "streams":
        streams = _log_int(rng, 2, 128)
        case.update(streams=streams, slots=next(s for s in (4, 8, 32, 128) if s >= streams),
                    draft_len=rng.choice([1, 2, 3, 3]))
    else:
        model, dtype = rng.choice([("mcd", "bf16"), ("mcd", "bf16"), ("mcd", "int8"), ("tiny", "f32"), ("tiny", "bf16")])
        case.update(model=model, dtype=dtype, draft_len=rng.randint(0, 7 if model == "mcd" else 3),
                    host=rng.random() < 0.4)
    return case


# ---- models --------------------------------------------------------------------------------
_kept = {}


def _keep(key, make):
    if key not in _kept:
        _kept[key] = make()
    return _kept[key]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _config(case, **kw):
    base = synth.TINY.replace(temperature=0.9) if case["model"] == "tiny" else synth.MCD
    dtype = {"f32": synth.WEIGHT_F32, "bf16": synth.WEIGHT_BF16, "int8": synth.WEIGHT_INT8}[case["dtype"]]
    return base.replace(weight_dtype=dtype, draft_len=case["draft_len"], max_streams=case["slots"],
                        draft_mode=synth.DRAFT_TREE if case["nodes"] else synth.DRAFT_SAMPLE, **kw)


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(seed)


def _gaussian(gen, shape, std):
    return torch.randn(shape, generator=gen, device=_device()) * std


def _stored(t, dtype):
    """The values of a tensor in the weights' type, as fp32."""
    return t if dtype == synth.WEIGHT_F32 else t.to(torch.bfloat16).float()


def _host(t, dtype):
    """What the binding takes: fp32 arrays, or bf16 bit patterns."""
    if dtype == synth.WEIGHT_F32:
        return t.float().cpu().numpy()
    return t.to(torch.bfloat16).view(torch.int16).cpu().numpy().view(np.uint16)


def _shift(first, last):
    """How far a code at position `first` is from the code it predicts at `last`."""
    return SHIFT * sum(range(first + 1, last + 1))


def _layers(gen, c, scale=1.0):
    """Random transformer layers; `scale` is that of the two products that write the residual
    stream (a row's own embedding stays its largest part)."""
    D, out = c.head_dim, {}
    for l in range(c.n_layers):
        for name, shape, std in (("wq", (c.n_q_heads * D, c.hidden), 0.02), ("wk", (c.n_kv_heads * D, c.hidden), 0.02),
                                 ("wv", (c.n_kv_heads * D, c.hidden), 0.02),
                                 ("wo", (c.hidden, c.n_q_heads * D), 0.02 * scale),
                                 ("wg", (c.ffn, c.hidden), 0.02), ("wu", (c.ffn, c.hidden), 0.02),
                                 ("wd", (c.hidden, c.ffn), 0.02 * scale)):
            out[f"layers.{l}.{name}"] = _gaussian(gen, shape, std)
        for name, n in (("attn_norm", c.hidden), ("ffn_norm", c.hidden), ("q_norm", D), ("k_norm", D)):
            out[f"layers.{l}.{name}"] = 1 + _gaussian(gen, (n,), 0.1)
    out["final_norm"] = 1 + _gaussian(gen, (c.hidden,), 0.1)
    return out


def _mcd_weights(cfg, tree):
    gen = _generator(11)
    w = _layers(gen, cfg, 1 / math.sqrt(2 * cfg.n_layers))
    V, H, P = cfg.vocab, cfg.hidden, cfg.n_pos
    rows = max(V, cfg.c0_vocab)
    table = [_gaussian(gen, (rows if i == 0 else V, H), 1.0) for i in range(P)]
    odd = (torch.arange(V, device=table[0].device) % 2 == 1)[:, None]
    for i, t in enumerate(table):
        w[f"embed.{i}"] = t
    for s in range(1, P + 1):
        head = _gaussian(gen, (V, H), 0.02)
        gain = PEAK / (0.93 * H)
        for lag in range(1, min(s, cfg.draft_len + 1) + 1):
            e, by = table[s - lag][:V], _shift(s - lag, s)
            for r, strength in enumerate(RANKS if tree else RANKS[:1]):
                part = torch.roll(e, by + r * SIBLING, 0)
                if r == 0 and lag > 2:
                    part = torch.roll(e * ~odd, by, 0) + torch.roll(e * odd, by + WRONG, 0)
                head += gain * strength * part
        w[f"head.{s}"] = head
    for j in range(1, max(cfg.draft_len, 1) + 1):
        w[f"offset.{j}"] = _gaussian(gen, (H,), 0.02)
    return {k: _stored(v, cfg.weight_dtype) for k, v in w.items()}


def _outer_config():
    return synth.OUTER.replace(text_vocab=2 * synth.OUTER.c0_vocab, prompt_len=512, frames=33)


def _outer_weights(cfg, inner):
    """The CodeDecoder: a row's text token predicts its c0."""
    gen = _generator(13)
    w = _layers(gen, cfg)
    text = _gaussian(gen, (cfg.text_vocab, cfg.hidden), 6.0)
    pairs = text.view(2, cfg.c0_vocab, cfg.hidden).sum(0)
    w["text_embed"] = text
    w["c0_head"] = _gaussian(gen, (cfg.c0_vocab, cfg.hidden), 0.02) + PEAK / (0.77 * 6.0 * cfg.hidden) * pairs
    w["c0_embed"] = _gaussian(gen, (cfg.c0_vocab, cfg.hidden), 1.0)
    w[f"code_embed.{inner.n_pos}"] = _gaussian(gen, (inner.vocab, cfg.hidden), 1.0)
    return {k: _stored(v, cfg.weight_dtype) for k, v in w.items()}


def _tree(nodes):
    """`nodes` nodes in breadth-first order: four candidates below the first row, then four
    below each node of the depth before, best ranks first."""
    parent, rank, level, depth = [], [], [-1], 1
    while len(parent) < nodes and depth <= TREE_DEPTH:
        start = len(parent)
        left = nodes - len(parent) if depth == TREE_DEPTH else min(nodes - len(parent), 4 if depth == 1 else 12)
        spread = sorted((r, p) for p in level for r in range(len(RANKS)))[:left]
        for r, p in sorted(spread, key=lambda rp: (rp[1], rp[0])):
            parent.append(p)
            rank.append(r)
        level, depth = list(range(start, len(parent))), depth + 1
    return parent, rank


def _decoder(case):
    cfg = _config(case)
    key = ("decoder", cfg, case["nodes"])

    def make():
        w = _mcd_weights(cfg, case["nodes"] > 0)
        dec = mcd.Decoder(cfg, {k: _host(v, cfg.weight_dtype) for k, v in w.items()})
        if case["nodes"]:
            mcd.mcd_set_tree(dec.ctx, *_tree(case["nodes"]))
        return dec

    return cfg, _keep(key, make)


def _pipeline():
    def make():
        inner, outer = synth.PIPE_INNER, _outer_config()
        iw, ow = _mcd_weights(inner, False), _outer_weights(outer, inner)
        return mcd.Pipeline(outer, inner, {k: _host(v, outer.weight_dtype) for k, v in ow.items()},
                            {k: _host(v, inner.weight_dtype) for k, v in iw.items()})

    return _keep("pipeline", make)


# ---- states and passes -----------------------------------------------------------------------
def _frame_inputs(cfg, case, seed):
    gen = _generator(seed)
    n = case["streams"]
    cond = _gaussian(gen, (n, cfg.hidden), 1.0)
    c0 = torch.randint(0, max(cfg.c0_vocab, cfg.vocab), (n,), generator=gen, device=cond.device, dtype=torch.int32)
    return cond, c0


def _prompt(case, seed):
    """Text ids of the prompt, then for every later row its text id and the codes before it."""
    outer, inner = _outer_config(), synth.PIPE_INNER
    gen, dev = _generator(seed), _device()
    ids = torch.randint(0, outer.text_vocab, (case["tokens"],), generator=gen, device=dev, dtype=torch.int32)
    rows = case.get("rows", 0)
    text = torch.randint(0, outer.text_vocab, (rows,), generator=gen, device=dev, dtype=torch.int32)
    codes = torch.randint(0, inner.vocab, (rows, inner.n_pos + 1), generator=gen, device=dev, dtype=torch.int32)
    return ids, text, codes


def _gemm_inputs(case, seed):
    gen = _generator(seed)
    a = _gaussian(gen, (case["m"], case["k"]), 0.02).to(torch.bfloat16)
    b = _gaussian(gen, (case["n"], case["k"]), 1.0).to(torch.bfloat16)
    return a, b


def _aligned(nbytes):
    """A device buffer that starts on a 1024-byte boundary, as the laid-out operands have to."""
    raw = torch.empty(nbytes + 1024, dtype=torch.uint8, device="cuda")
    off = -raw.data_ptr() % 1024
    return raw[off:off + nbytes]


def prepare(case, seed):
    kind, s = case["kind"], {"kind": case["kind"], "case": case}
    if kind == "topk":
        gen, n, k = _generator(seed), case["rows"], case["top_k"]
        s.update(logits=_gaussian(gen, (n, case["vocab"]), 2.0),
                 ids=torch.zeros((n, k), dtype=torch.int32, device="cuda"),
                 weights=torch.zeros((n, k), dtype=torch.int32, device="cuda"),
                 sums=torch.zeros((n,), dtype=torch.int64, device="cuda"), stream=torch.cuda.current_stream())
    elif kind == "gemm":
        a, b = _gemm_inputs(case, seed)
        s.update(b=b, a_tiled=_aligned(a.numel() * 2), b_tiled=_aligned(b.numel() * 2), stream=torch.cuda.current_stream(),
                 y=torch.zeros((case["n"], case["m"]), device="cuda"), err=torch.zeros((1,), dtype=torch.int32, device="cuda"))
        mcd.mcd_tc_tile(case["m"], case["k"], a, s["a_tiled"], s["stream"])
        torch.cuda.synchronize()
    elif kind == "frame":
        cfg, dec = _decoder(case)
        cond, c0 = _frame_inputs(cfg, case, seed)
        n = case["streams"]
        if cfg.c0_vocab:
            emb = None
        else:   # the model takes the c0 embedding itself
            emb = _keep(("c0 table", cfg), lambda: _mcd_weights(cfg, case["nodes"] > 0)["embed.0"])[c0.long()].contiguous()
            c0 = None
        trace = torch.zeros(mcd.mcd_trace_bytes(dec.ctx), dtype=torch.uint8, device="cuda")
        codes = torch.zeros((n, cfg.n_pos), dtype=torch.int32, device="cuda")
        stats = torch.zeros((n, 8), dtype=torch.int32, device="cuda")
        if case["host"]:
            cond, c0, emb, codes, stats = (None if t is None else t.cpu().pin_memory() for t in (cond, c0, emb, codes, stats))
        s.update(ctx=dec.ctx, cond=cond, c0=c0, emb=emb, trace=trace, codes=codes, stats=stats, ids=list(range(n)),
                 out=dict(_trace_views(cfg, case, trace), codes=codes, stats=stats))
    else:
        pipe, outer = _pipeline(), _outer_config()
        ids, text, codes = _prompt(case, seed)
        n = 1 + case.get("rows", 0)
        s.update(o=pipe.o, ids=ids, text=text.tolist(), codes=[c.contiguous() for c in codes],
                 trace=torch.zeros((n, mcd.mcd_outer_trace_floats(pipe.o)), device="cuda"),
                 c0=torch.zeros((n,), dtype=torch.int32, device="cuda"))
        s["c0_at"] = [s["c0"][i:] for i in range(n)]
    return s


def _trace_views(cfg, case, trace):
    """The logits of a frame's trace: every call's verify and draft rows of every stream."""
    n, V = case["streams"], cfg.vocab
    per = trace.numel() // case["slots"]
    f = trace.view(case["slots"], per)[:n]
    head = mcd.CALL_TRACE_DTYPE.itemsize * mcd.MAX_CALLS
    size = mcd.MAX_CALLS * mcd.MAX_ROWS * V * 4
    part = lambda at, nbytes: f[:, at:at + nbytes].view(torch.float32)  # noqa: E731
    if not case["nodes"]:
        return {"verify": part(head, size), "draft": part(head + size, size)}
    at = head + 2 * size + mcd.TREE_TRACE_DTYPE.itemsize * mcd.MAX_CALLS
    return {"draft": part(head + size, size), "verify": part(at, mcd.MAX_CALLS * mcd.MAX_TREE_ROWS * V * 4)}


def run(s):
    kind, c = s["kind"], s["case"]
    if kind == "topk":
        mcd.mcd_topk_softmax_static(c["rows"], c["vocab"], c["top_k"], 0.9, s["logits"], s["ids"], s["weights"], s["sums"],
                                    s["stream"])
        return {"ids": s["ids"], "weights": s["weights"], "sums": s["sums"]}
    if kind == "gemm":
        mcd.mcd_tc_tile(c["n"], c["k"], s["b"], s["b_tiled"], s["stream"])
        mcd.mcd_tc_gemm_tiled(c["m"], c["n"], c["k"], 0, s["a_tiled"], s["b_tiled"], s["y"], s["err"], s["stream"])
        return {"y": s["y"], "err": s["err"]}
    if kind == "frame":
        mcd.mcd_set_trace(s["ctx"], s["trace"])
        if c["host"]:
            mcd.mcd_decode_frame_host(s["ctx"], 0, 0, s["cond"], s["c0"], s["emb"], s["codes"], s["stats"])
        elif c["slots"] == 1:
            mcd.mcd_decode_frame(s["ctx"], 0, 0, s["cond"], s["c0"], s["emb"], s["codes"], s["stats"])
        else:
            mcd.mcd_decode_frames(s["ctx"], s["ids"], s["ids"], s["cond"], s["c0"], s["emb"], s["codes"], s["stats"])
        return s["out"]
    mcd.mcd_outer_set_trace(s["o"], s["trace"], len(s["c0_at"]))
    mcd.mcd_outer_prefill(s["o"], 0, s["ids"], s["c0_at"][0])
    for f, (codes, text) in enumerate(zip(s["codes"], s["text"])):
        mcd.mcd_outer_step(s["o"], codes, text, s["c0_at"][f + 1])
    return {"logits_cond_emb": s["trace"], "c0": s["c0"]}


# ---- what a pass cannot do without -----------------------------------------------------------
def _layer_params(c):
    D = c.head_dim
    return c.hidden * (2 * c.n_q_heads * D + 2 * c.n_kv_heads * D + 3 * c.ffn)


def work(case):
    if case["kind"] == "topk":
        n, V, k = case["rows"], case["vocab"], case["top_k"]
        return {"bytes": n * (4 * V + 8 * k + 8), "flops": 2 * n * V}
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2 * k * (m + n) + 4 * m * n, "flops": 2 * m * n * k}
    if case["kind"] == "frame":
        # the backbone once per call of the slowest stream, the LM heads its rows read, the
        # logits that come back
        c, K = _config(case), case["draft_len"]
        per = {"f32": 4, "bf16": 2, "int8": 1}[case["dtype"]]
        tokens = 1 + (1 if K else 0) + sum(0.5 ** (j - 1) for j in range(2, K + 1))
        calls = 1 + math.ceil((c.n_pos - 1) / tokens)
        rows = 1 + (case["nodes"] or K)
        heads = min(c.n_pos, 1 + 2 * K)
        body = c.n_layers * _layer_params(c)
        out = 4 * case["streams"] * c.vocab * (rows + K)
        per_row = 2 * (body + (1 + K) * c.vocab * c.hidden)
        return {"bytes": calls * (per * (body + heads * c.vocab * c.hidden) + out),
                "flops": calls * case["streams"] * rows * per_row}
    c = _outer_config()
    body, head = c.n_layers * _layer_params(c), c.c0_vocab * c.hidden
    kv = 2 * 2 * c.n_layers * c.n_kv_heads * c.head_dim
    T, R = case["tokens"], case.get("rows", 0)
    at = sum(T + i for i in range(R))
    scores = 4 * c.n_layers * c.n_q_heads * c.head_dim
    return {"bytes": (1 + R) * 2 * (body + head) + kv * (T + at + R) + 2 * c.hidden * (T + 17 * R),
            "flops": 2 * body * (T + R) + 2 * head * (1 + R) + scores * (T * T // 2 + at)}


# About four times what another order of the sums shows (the persistent kernels add partial
# sums with atomics, so the same pass twice is one) and what exact() shows, the larger.
def tolerance(case):
    if case["kind"] == "topk":
        return "exact"
    if case["kind"] == "gemm":
        return {"rel": 4e-6, "max": 1e-4}          # fp32 sums of exact bf16 products
    if case["kind"] in ("prefill", "rows"):
        return {"rel": 2e-3, "max": 5e-2}          # K / V and the prompt's operands in bf16
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 2e-5}
    if case["streams"] > 4 or case["nodes"] > 15:
        return {"rel": 5e-3, "max": 0.1}           # one bf16 operand in places
    return {"rel": 1e-5, "max": 3e-4}              # bf16 hi + lo operands: about 16 bits


# ---- the same in 64 bits ---------------------------------------------------------------------
def _quantised(w):
    """Per-row 8-bit weights: s = fp32(max |w| / 127), q = round(w / s)."""
    s = w.abs().amax(1, keepdim=True) / torch.full((1, 1), 127.0, device=w.device)   # an IEEE division
    return torch.where(s > 0, torch.clamp(torch.round(w / s), -127, 127).double() * s.double(), torch.zeros((), device=w.device, dtype=torch.float64))


def _values(w, dtype):
    """64-bit values of the weights a context computes with."""
    streamed = ("wq", "wk", "wv", "wo", "wg", "wu", "wd")
    q8 = dtype == synth.WEIGHT_INT8
    return {k: _quantised(v) if q8 and (k.split(".")[-1] in streamed or k.startswith("head.")) else v.double()
            for k, v in w.items()}


def _rms(x, gain, eps):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * gain


def _forward(c, w, x, cache_bf16=False):
    """Post-norm hidden states of sequences x [B, T, H] (causal, positions 0..T-1)."""
    B, T, _ = x.shape
    D, hq, hk = c.head_dim, c.n_q_heads, c.n_kv_heads
    ang = torch.arange(T, device=x.device, dtype=torch.float64)[:, None] * torch.pow(
        torch.tensor(c.rope_base, dtype=torch.float64, device=x.device), -2.0 * torch.arange(D // 2, device=x.device, dtype=torch.float64) / D)
    cos, sin = ang.cos(), ang.sin()

    def rope(v):
        a, b = v[..., :D // 2], v[..., D // 2:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

    mask = torch.full((T, T), -math.inf, device=x.device, dtype=torch.float64).triu(1)
    for l in range(c.n_layers):
        p = f"layers.{l}."
        n = _rms(x, w[p + "attn_norm"], c.rms_eps)
        q, k, v = ((n @ w[p + m].T).view(B, T, -1, D).transpose(1, 2) for m in ("wq", "wk", "wv"))
        q, k = rope(_rms(q, w[p + "q_norm"], c.rms_eps)), rope(_rms(k, w[p + "k_norm"], c.rms_eps))
        if cache_bf16:
            k, v = (t.float().to(torch.bfloat16).double() for t in (k, v))
        k, v = (t.repeat_interleave(hq // hk, 1) for t in (k, v))
        a = torch.softmax(q @ k.transpose(-1, -2) / math.sqrt(D) + mask, -1) @ v
        x = x + a.transpose(1, 2).reshape(B, T, hq * D) @ w[p + "wo"].T
        n = _rms(x, w[p + "ffn_norm"], c.rms_eps)
        x = x + (torch.nn.functional.silu(n @ w[p + "wg"].T) * (n @ w[p + "wu"].T)) @ w[p + "wd"].T
    return _rms(x, w["final_norm"], c.rms_eps)


def _last_hidden(cfg, w, cond, seqs):
    """Hidden state of the last position of [cond[s], E_0(t_0), E_1(t_1), ...] for (s, t) in seqs."""
    T = 1 + max(len(t) for _, t in seqs)
    x = torch.zeros((len(seqs), T, cfg.hidden), device=cond.device, dtype=torch.float64)
    x[:, 0] = cond[[s for s, _ in seqs]]
    for i in range(T - 1):
        at = [(n, t[i]) for n, (_, t) in enumerate(seqs) if len(t) > i]
        x[[n for n, _ in at], i + 1] = w[f"embed.{i}"][[t for _, t in at]]
    h = torch.cat([_forward(cfg, w, part) for part in x.split(64)])
    return h[torch.arange(len(seqs), device=h.device), [len(t) for _, t in seqs]]


def _exact_frames(case, seed):
    """Every call of every stream's frame.  The predicted codes hold all the probability a
    draw can reach, so a row's largest logit is what it emits or drafts."""
    cfg = _config(case)
    w = _values(_mcd_weights(cfg, case["nodes"] > 0), cfg.weight_dtype)
    cond, c0 = _frame_inputs(cfg, case, seed)
    cond, P, K, V, n_s = cond.double(), cfg.n_pos, cfg.draft_len, cfg.vocab, case["streams"]
    parent, rank = _tree(case["nodes"]) if case["nodes"] else (list(range(-1, K - 1)), [0] * K)
    depth = []
    for i, p in enumerate(parent):
        depth.append(1 if p < 0 else depth[p] + 1)
    deepest = max(depth, default=0)
    width = mcd.MAX_TREE_ROWS if case["nodes"] else mcd.MAX_ROWS
    verify = torch.zeros((n_s, mcd.MAX_CALLS, width, V), dtype=torch.float64, device=cond.device)
    draft = torch.zeros((n_s, mcd.MAX_CALLS, mcd.MAX_ROWS, V), dtype=torch.float64, device=cond.device)
    codes = [[int(v)] for v in c0.tolist()]
    cand = [[] for _ in range(n_s)]                # [depth - 1][rank] codes drafted for the next call
    for call in range(P):
        live = [s for s in range(n_s) if len(codes[s]) <= P]
        if not live:
            break
        rows = []                                   # (stream, node, codes fed up to the row)
        for s in live:
            a, path = len(codes[s]) - 1, {-1: []}
            rows.append((s, -1, list(codes[s])))
            for i, p in enumerate(parent):
                if depth[i] <= len(cand[s]) and a + depth[i] < P:
                    path[i] = path[p] + [cand[s][depth[i] - 1][rank[i]]]
                    rows.append((s, i, codes[s] + path[i]))
        h = _last_hidden(cfg, w, cond, [(s, t) for s, _, t in rows])
        at = {(s, node): n for n, (s, node, _) in enumerate(rows)}
        top = [0] * len(rows)
        for pos in {len(t) for _, _, t in rows}:
            group = [n for n, (_, _, t) in enumerate(rows) if len(t) == pos]
            z = h[group] @ w[f"head.{pos}"].T
            for n, zi, best in zip(group, z, z.argmax(1).tolist()):
                s, node, _ = rows[n]
                verify[s, call, 1 if call == 0 else node + 1] = zi
                top[n] = best
        ask = {}
        for s in live:
            node, a, best, emit = -1, len(codes[s]) - 1, top[at[s, -1]], []
            n = at[s, -1]
            while True:
                emit.append(best)
                kept = [i for i, p in enumerate(parent) if p == node and depth[i] <= len(cand[s]) and a + depth[i] <= P
                        and cand[s][depth[i] - 1][rank[i]] == best]
                if not kept or (s, kept[0]) not in at:
                    break
                node = kept[0]
                n = at[s, node]
                best = top[n]
            codes[s] = codes[s] + emit
            cand[s] = []
            for j in range(1, min(deepest, P - (len(codes[s]) - 1)) + 1):
                ask.setdefault((len(codes[s]) - 1 + j, j), []).append((s, n))
        for (pos, j), who in sorted(ask.items(), key=lambda kv: kv[0][1]):
            z = (h[[n for _, n in who]] + w[f"offset.{j}"]) @ w[f"head.{pos}"].T
            order = z.topk(len(RANKS), 1).indices.tolist()
            for (s, _), zi, best in zip(who, z, order):
                draft[s, call, j - 1] = zi
                cand[s].append(best)
    flat = lambda t: t.reshape(n_s, -1)  # noqa: E731
    return {"verify": flat(verify), "draft": flat(draft), "codes": None, "stats": None}


def _exact_rows(case, seed):
    cfg, inner = _outer_config(), synth.PIPE_INNER
    w = _values(_outer_weights(cfg, inner), cfg.weight_dtype)
    tables = {k: v.double() for k, v in _mcd_weights(inner, False).items() if k.startswith("embed.")}
    ids, text, codes = _prompt(case, seed)
    rows = w["text_embed"][text.long()] + w["c0_embed"][codes[:, 0].long()] + w[f"code_embed.{inner.n_pos}"][codes[:, -1].long()]
    for j in range(1, inner.n_pos):
        rows = rows + tables[f"embed.{j}"][codes[:, j].long()]
    h = _forward(cfg, w, torch.cat([w["text_embed"][ids.long()], rows])[None], cache_bf16=True)[0, case["tokens"] - 1:]
    z = h @ w["c0_head"].T
    return {"logits_cond_emb": torch.cat([z, h, w["c0_embed"][z.argmax(1)]], 1), "c0": None}


def exact(case, seed):
    if case["kind"] == "topk":
        return None                                # whole numbers: they are the same or wrong
    if case["kind"] == "gemm":
        a, b = _gemm_inputs(case, seed)
        return {"y": b.double() @ a.double().T, "err": None}
    return _exact_frames(case, seed) if case["kind"] == "frame" else _exact_rows(case, seed)
