"""The work this framework is used for, as cases that can be timed and compared: decode steps over short and
long caches, single sequences and ragged batches, with direct calls and as a captured graph; a selection that is
reused for an interval; dense attention for the first decode token; prompt ingestion; the importance-query
predictor; and whole requests that run through every entry point.

A case is a dict of plain values.  `kind` says which pass it is:

  step     decode steps over a filled cache: per producer group of four layers one selection, then attention layer
           by layer; `interval` consecutive steps, the first of which refreshes the lists (interval 1 = one step)
  dense    the same schedule under the dense rule (first decode token): attention over every cached token
  prefill  an empty sequence slot takes a prompt: K/V rows appended layer by layer, then all keys projected
  predict  the predictor forward of `producers` producer layers, one hidden state per decoding sequence
  request  prompts appended and projected, then `steps` decode steps: append, deferred projection, predictor,
           selection, attention

Shapes are those of an 8B model (32 query heads, 8 KV heads, head dimension 128) unless a case says otherwise."""
import math

import numpy as np
import torch

from paper_2503_07518_b200 import binding as tb

HEAD_DIM = 128
GROUP_LAYERS = 4            # consumer layers of one producer
DTYPES = {"bf16": tb.TB_BF16, "fp32": tb.TB_F32}
SCOPES = {"kv_head": tb.TB_SCOPE_KV_HEAD, "q_head": tb.TB_SCOPE_Q_HEAD, "layer": tb.TB_SCOPE_LAYER}
NMODES = {"dilate": tb.TB_NEIGHBOR_DILATE, "cluster": tb.TB_NEIGHBOR_CLUSTER}
REDUCES = {"sum": tb.TB_GROUP_SUM, "max": tb.TB_GROUP_MAX}

_STEP = dict(kind="step", dtype="bf16", layers=8, batch=1, len_lo=32768, len_hi=32768, q_heads=32, kv_heads=8, imp_dim=32,
             budget=1024, sinks=0, recent=0, radius=0, nmode="dilate", interval=1, scope="kv_head", reduce="sum",
             outliers=0, planted=0, lists=False, graph=False)
_PREFILL = dict(kind="prefill", dtype="bf16", layers=4, batch=1, len_lo=32768, len_hi=32768, q_heads=32, kv_heads=8, imp_dim=32,
                scope="kv_head", outliers=4)
_PREDICT = dict(kind="predict", dtype="bf16", tokens=1, producers=8, model_dim=4096, hidden_dim=512, slots=4, q_heads=32,
                imp_dim=32)
_REQUEST = dict(kind="request", dtype="bf16", layers=4, batch=4, len_lo=1000, len_hi=2100, q_heads=32, kv_heads=8, imp_dim=16,
                budget=192, sinks=16, recent=32, radius=1, nmode="cluster", interval=4, scope="kv_head", reduce="sum",
                outliers=4, planted=0, steps=16, model_dim=4096, hidden_dim=512)


def listed():
    return [
        # the smallest call: one layer, fp32, 4K tokens, each step called directly -- latency and launches
        dict(_STEP, name="step_4k_fp32", dtype="fp32", layers=1, q_heads=8, len_lo=4096, len_hi=4096, budget=256, sinks=4,
             recent=64, lists=True),
        # a few short chats decoded together, called directly: host path and launches, odd lengths, narrow projection
        dict(_STEP, name="step_chats", layers=16, batch=3, len_lo=700, len_hi=3100, imp_dim=16, budget=300, sinks=16, recent=64,
             outliers=4),
        # a whole decode step of a 32-layer model at 32K tokens, 10 % budget, captured once and replayed
        dict(_STEP, name="step_32k", layers=32, budget=3276, outliers=4, graph=True),
        # batched serving: 16 sequences of 8K to 16K tokens
        dict(_STEP, name="step_batch16", batch=16, len_lo=8192, len_hi=16384, budget=1024),
        # long context at batch 1 with sinks, a recent window and needles that outscore everything else
        dict(_STEP, name="step_128k", len_lo=131072, len_hi=131072, budget=2048, sinks=16, recent=256, planted=64, graph=True),
        # a prediction interval: one refresh with +-1 neighbours, fifteen steps that reuse its lists
        dict(_STEP, name="interval_64k", layers=4, batch=8, len_lo=65536, len_hi=65536, budget=3276, recent=16, radius=1,
             interval=16),
        # one list per query head, cluster neighbours
        dict(_STEP, name="step_per_head", layers=4, batch=2, len_lo=15000, len_hi=25000, budget=777, sinks=4, recent=64, radius=1,
             nmode="cluster", scope="q_head", lists=True),
        # the first decode token after the prompt: dense attention
        dict(_STEP, name="dense_16k", kind="dense", batch=2, len_lo=14000, len_hi=16384, budget=1, outliers=4),
        # a 32K prompt enters the caches
        dict(_PREFILL, name="prefill_32k"),
        # query prediction for a single decoding sequence, and for a batch of them
        dict(_PREDICT, name="predict_1"),
        dict(_PREDICT, name="predict_24", tokens=24),
        # four requests from their prompts through sixteen decoded tokens: every entry point, small calls
        dict(_REQUEST, name="request_short"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        c = _draw_any(rng)
        if _affordable(c):
            return c


def _draw_any(rng):
    kind = rng.choice(["step"] * 9 + ["dense"] * 2 + ["prefill"] * 3 + ["predict"] * 3 + ["request"] * 3)
    dtype = "fp32" if rng.random() < 0.15 else "bf16"
    if kind == "predict":
        return dict(_PREDICT, dtype=dtype, tokens=_log_int(rng, 1, 64), producers=rng.choice([1, 2, 4, 8]),
                    model_dim=32 * _log_int(rng, 32, 160), hidden_dim=rng.choice([256, 512, 1024]), slots=rng.choice([1, 3, 4]),
                    q_heads=rng.choice([8, 16, 32]), imp_dim=rng.choice([16, 32]))
    q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (32, 8), (8, 8), (16, 8), (16, 4), (28, 4), (32, 4)])
    shape = dict(dtype=dtype, q_heads=q_heads, kv_heads=kv_heads, imp_dim=rng.choice([16, 32, 32]), outliers=rng.choice([0, 4]))
    scope = rng.choice(["kv_head"] * 6 + ["q_head", "layer"])
    hi = _log_int(rng, 512, 131072) if kind != "request" else _log_int(rng, 256, 8192)
    lo = max(64, int(hi * rng.uniform(0.4, 1.0)))
    if kind == "prefill":
        return dict(_PREFILL, **shape, scope=scope, layers=rng.choice([1, 2, 4, 8]), batch=_log_int(rng, 1, 16), len_lo=lo, len_hi=hi)
    select = dict(shape, scope=scope, len_lo=lo, len_hi=hi, budget=max(16, int(hi * math.exp(rng.uniform(math.log(0.015), math.log(0.2))))),
                  sinks=rng.choice([0, 4, 16, 128]), recent=rng.choice([0, 16, 64, 256]), radius=rng.choice([0, 0, 0, 1]),
                  nmode=rng.choice(["dilate", "cluster"]), interval=rng.choice([1, 1, 1, 4, 16]),
                  reduce=rng.choice(["sum"] * 5 + ["max"]) if scope == "kv_head" else "sum")
    if kind == "request":
        select.update(recent=rng.choice([16, 64]), interval=rng.choice([1, 4, 16]))
        return dict(_REQUEST, **select, layers=rng.choice([2, 4, 8]), batch=_log_int(rng, 1, 16), steps=rng.choice([8, 16]))
    if kind == "dense":
        return dict(_STEP, **dict(select, budget=1, interval=1, radius=0, scope="kv_head", reduce="sum", sinks=0, recent=0), **{
            "kind": "dense", "layers": rng.choice([1, 4, 8]), "batch": _log_int(rng, 1, 16), "graph": rng.random() < 0.4})
    if select["interval"] > 1:
        select["recent"] = max(16, select["recent"])
    planted = 64 if scope == "kv_head" and hi >= 16384 and rng.random() < 0.3 else 0
    return dict(_STEP, **select, layers=rng.choice([1, 4, 8, 16, 32]), batch=_log_int(rng, 1, 32), planted=planted,
                graph=rng.random() < 0.4, lists=rng.random() < 0.3)


def _affordable(c):
    """No larger than the listed cases in memory, traffic and calls."""
    if c["kind"] == "predict":
        return True
    kv = c["layers"] * sum(_lengths(c)) * c["kv_heads"] * 2 * HEAD_DIM * _es(c)
    calls = c["layers"] * (c["interval"] if c["kind"] == "step" else c.get("steps", 1) * 3)
    return kv <= 9e9 and calls <= 256 and work(c)["bytes"] <= 2e10


# ---- sizes ------------------------------------------------------------------------------------------

def _es(c):
    return 2 if c["dtype"] == "bf16" else 4


def _lengths(c):
    """Tokens per sequence: a ragged batch between the case's bounds (the longest is the upper one)."""
    if c["batch"] == 1 or c["len_lo"] == c["len_hi"]:
        return [c["len_hi"]] * c["batch"]
    r = np.random.RandomState((c["len_lo"] * 7919 + c["len_hi"] * 31 + c["batch"]) % (1 << 31))
    return [c["len_hi"]] + [int(x) for x in r.randint(c["len_lo"], c["len_hi"] + 1, size=c["batch"] - 1)]


def _heads(c):
    """Key streams, lists and attention units per (layer, sequence), importance queries per list's token."""
    hi = 1 if c["scope"] == "layer" else c["kv_heads"]
    hl = {"kv_head": c["kv_heads"], "q_head": c["q_heads"], "layer": 1}[c["scope"]]
    return hi, hl, max(hl, c["kv_heads"]), (1 if c["scope"] == "layer" else c["q_heads"])


def _rows(c, L):
    """Expected distinct cache rows that one KV head's query heads attend to."""
    if c["kind"] == "dense":
        return L
    s = min(c["sinks"], L)
    n = max(0, L - c["recent"] - s)
    k = min(c["budget"], n)
    if n and k < n:
        spread = 1
        if c["radius"]:
            spread = 1 + 2 * c["radius"] if c["nmode"] == "dilate" else 1 + c["radius"]
        if c["scope"] == "q_head":
            spread *= c["q_heads"] // c["kv_heads"]
        k = n * (1.0 - (1.0 - k / n) ** spread)
    return s + k + (L - s - n)


def _select_work(c, lengths):
    hi, hl, _, nq = _heads(c)
    cand = sum(max(0, L - c["sinks"] - c["recent"]) for L in lengths)
    return cand * hi * c["imp_dim"] * _es(c) + len(lengths) * nq * c["imp_dim"] * 4, 2.0 * cand * hl * c["imp_dim"]


def _attend_work(c, lengths):
    rows = sum(_rows(c, L) for L in lengths)
    io = len(lengths) * c["q_heads"] * HEAD_DIM * (_es(c) + 4)
    return rows * c["kv_heads"] * 2 * HEAD_DIM * _es(c) + io, 4.0 * rows * c["q_heads"] * HEAD_DIM


def _append_work(c, tokens):
    hi = _heads(c)[0]
    io = tokens * c["kv_heads"] * 2 * HEAD_DIM * _es(c)
    return 2 * io + tokens * hi * c["imp_dim"] * _es(c), 2.0 * tokens * c["kv_heads"] * HEAD_DIM * c["imp_dim"]


def _predict_work(c, tokens, slots):
    n_out = slots * (c["q_heads"] if c.get("scope", "kv_head") != "layer" else 1) * c["imp_dim"]
    weights = c["hidden_dim"] * (c["model_dim"] + n_out) + 2 * c["model_dim"]
    return (weights + tokens * c["model_dim"]) * _es(c) + tokens * n_out * 4, 2.0 * tokens * c["hidden_dim"] * (c["model_dim"] + n_out)


def work(case):
    c = case
    parts = []
    if c["kind"] == "predict":
        parts.append((c["producers"],) + _predict_work(c, c["tokens"], c["slots"]))
    else:
        lengths = _lengths(c)
        if c["kind"] in ("prefill", "request"):
            parts.append((c["layers"],) + _append_work(c, sum(lengths)))
        if c["kind"] == "step":
            parts.append((c["layers"],) + _select_work(c, lengths))
        if c["kind"] in ("step", "dense"):
            parts.append((c["layers"] * c["interval"],) + _attend_work(c, lengths))
        if c["kind"] == "request":
            for t in range(c["steps"]):
                now = [L + t + 1 for L in lengths]
                parts.append((c["layers"],) + _append_work(c, len(now)))
                if t % c["interval"] == 0:
                    parts.append((len(_groups(c)),) + _predict_work(c, len(now), GROUP_LAYERS))
                    parts.append((c["layers"],) + _select_work(c, now))
                parts.append((c["layers"],) + _attend_work(c, now))
    return {"bytes": float(sum(n * b for n, b, _ in parts)), "flops": float(sum(n * f for n, _, f in parts))}


def tolerance(case):
    """Inputs in the storage type, products accumulated in fp32.  Where a ranking is part of the pass, a correct
    implementation may order two tokens whose scores agree to fp32 rounding either way: one such swap changes a
    head's output by about 1 / sqrt(budget), and the entries of its list between the two positions."""
    if case["kind"] == "prefill":               # copied rows are exact, projected keys rounded once to the storage type
        return {"rel": 2e-3, "max": 1e-2} if case["dtype"] == "bf16" else {"rel": 1e-5}
    if case["kind"] == "predict":               # two fp32 products in a row; weights and states exact in the storage type
        return {"rel": 1e-4} if case["dtype"] == "bf16" else {"rel": 1e-5}
    if case["kind"] == "dense":
        return {"rel": 1e-4} if case["dtype"] == "bf16" else {"rel": 1e-5}
    return {"rel": 5e-3, "max": 0.5, "differ": 5e-3} if case["dtype"] == "bf16" else {"rel": 1e-5, "differ": 1e-3}


# ---- the passes -------------------------------------------------------------------------------------

def _groups(c):
    return [(l, min(GROUP_LAYERS, c["layers"] - l)) for l in range(0, c["layers"], GROUP_LAYERS)]


class State:
    """What a serving program keeps: the context (caches, lists), its inputs and output buffers."""


def _randn(gen, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=dtype)


def _keys_values(c, gen, tokens):
    """K and V rows of one layer, [tokens][kv heads][head dim]; a few key channels per head are large where the case asks."""
    dt = tb.torch_dtype(DTYPES[c["dtype"]])
    k, v = (_randn(gen, tokens, c["kv_heads"], HEAD_DIM, dtype=dt) for _ in range(2))
    if c["outliers"]:
        ch = torch.argsort(torch.rand(c["kv_heads"], HEAD_DIM, generator=gen, device="cuda"), dim=1)[:, :c["outliers"]]
        scale = torch.ones(c["kv_heads"], HEAD_DIM, device="cuda").scatter_(1, ch, 8.0)
        k.mul_(scale.to(dt))
    return k, v


def _context(c, gen, capacity):
    """An empty context with its key projections; the projections [layers][kv heads][head dim][d']."""
    radius = c.get("radius", 0)
    ctx = tb.Context(c["layers"], c["q_heads"], c["kv_heads"], HEAD_DIM, c["imp_dim"], DTYPES[c["dtype"]], c["batch"],
                     -(-capacity // 64) * 64, c.get("budget", 1), radius, list_scope=SCOPES[c["scope"]])
    W = (_randn(gen, c["layers"], c["kv_heads"], HEAD_DIM, c["imp_dim"]) / math.sqrt(HEAD_DIM)).to(tb.torch_dtype(DTYPES[c["dtype"]]))
    for l in range(c["layers"]):
        ctx.set_projection(l, W[l])
    return ctx, W


def _plant(c, gen, k, W, q_imp, lengths):
    """Raises `planted` random keys per sequence and KV head along the direction their importance query asks for."""
    start = 0
    for b, L in enumerate(lengths):
        q = q_imp[b].view(c["kv_heads"], -1, c["imp_dim"]).sum(1)
        d = torch.einsum("hcj,hj->hc", W.float(), q / q.norm(dim=1, keepdim=True)) * (2.0 * math.sqrt(c["imp_dim"]))
        pos = start + torch.randint(0, L, (c["kv_heads"], c["planted"]), generator=gen, device="cuda")
        for h in range(c["kv_heads"]):
            k[pos[h], h] += d[h].to(k.dtype)
        start += L


def _predictor(c, gen, slots, q_heads):
    dt = tb.torch_dtype(DTYPES[c["dtype"]])
    E, hid, n_out = c["model_dim"], c["hidden_dim"], slots * q_heads * c["imp_dim"]
    return dict(ln_weight=(1 + 0.1 * _randn(gen, E)).to(dt), ln_bias=(0.02 * _randn(gen, E)).to(dt),
                w1=(_randn(gen, hid, E) * E ** -0.5).to(dt), w2=(_randn(gen, n_out, hid) * 2.0 * hid ** -0.5).to(dt),
                dtype=DTYPES[c["dtype"]], n_q_heads=q_heads, n_slots=slots, imp_dim=c["imp_dim"])


def _hidden_states(c, gen, *shape):
    """Residual-stream-like hidden states: a shared offset and a few massive channels."""
    h = _randn(gen, *shape, c["model_dim"]) + 0.25
    h[..., torch.randint(0, c["model_dim"], (8,), generator=gen, device="cuda")] *= 20.0
    return h.to(tb.torch_dtype(DTYPES[c["dtype"]]))


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    s = State()
    s.c = c = case
    if c["kind"] == "predict":
        s.predictors = [_predictor(c, gen, c["slots"], c["q_heads"]) for _ in range(c["producers"])]
        s.hidden = _hidden_states(c, gen, c["producers"], c["tokens"])
        s.scratch = torch.empty(c["tokens"] * c["hidden_dim"], device="cuda")
        s.q_imp = torch.empty(c["producers"], c["slots"], c["tokens"], c["q_heads"], c["imp_dim"], device="cuda")
        return s
    s.lengths = lengths = _lengths(c)
    dt = tb.torch_dtype(DTYPES[c["dtype"]])
    _, hl, _, nq = _heads(c)
    B, layers = c["batch"], c["layers"]
    steps = c.get("steps", 0)
    s.ctx, W = _context(c, gen, max(lengths) + steps)
    s.zeros = [0] * B
    if c["kind"] in ("prefill", "request"):
        kv = [_keys_values(c, gen, sum(lengths)) for _ in range(layers)]
        s.k, s.v = [k for k, _ in kv], [v for _, v in kv]
        if c["kind"] == "prefill":
            s.out = [x[:, b, :, :L] for b, L in enumerate(lengths) for x in (s.ctx.kv, s.ctx.kimp)]
            return s
        s.k_new, s.v_new = (_randn(gen, steps, layers, B, c["kv_heads"], HEAD_DIM, dtype=dt) for _ in range(2))
        s.q = _randn(gen, steps, layers, B, c["q_heads"], HEAD_DIM, dtype=dt)
        s.ones = [1] * B
        s.predictors = [_predictor(c, gen, GROUP_LAYERS, nq) for _ in _groups(c)]
        refreshes = -(-steps // c["interval"])
        s.hidden = _hidden_states(c, gen, refreshes, len(s.predictors), B)
        s.scratch = torch.empty(B * c["hidden_dim"], device="cuda")
        s.q_imp = torch.empty(refreshes, len(s.predictors), GROUP_LAYERS, B, nq, c["imp_dim"], device="cuda")
        s.idx = torch.zeros(refreshes, layers, B, hl, s.ctx.index_capacity, dtype=torch.int32, device="cuda")
        s.cnt = torch.zeros(refreshes, layers, B, hl, dtype=torch.int32, device="cuda")
        s.out = torch.empty(steps, layers, B, c["q_heads"], HEAD_DIM, device="cuda")
        s.params = [_params(c, t) for t in range(steps)]
        projected = [L + (refreshes - 1) * c["interval"] + 1 for L in lengths]
        s.kimp = [s.ctx.kimp[:, b, :, :n] for b, n in enumerate(projected)]
        return s
    s.q = _randn(gen, c["interval"], layers, B, c["q_heads"], HEAD_DIM, dtype=dt)
    s.q_imp = _randn(gen, layers, B, nq, c["imp_dim"])
    for l in range(layers):
        k, v = _keys_values(c, gen, sum(lengths))
        if c["planted"]:
            _plant(c, gen, k, W[l], s.q_imp[l], lengths)
        s.ctx.append_kv(l, 1, None, lengths, k, v)
        del k, v
    s.ctx.project_keys(0, layers, None, s.zeros, lengths)
    s.out = torch.empty(c["interval"], layers, B, c["q_heads"], HEAD_DIM, device="cuda")
    s.idx = s.cnt = s.lse = None
    if c["lists"]:
        s.idx = torch.zeros(layers, B, hl, s.ctx.index_capacity, dtype=torch.int32, device="cuda")
        s.cnt = torch.zeros(layers, B, hl, dtype=torch.int32, device="cuda")
    if c["kind"] == "dense":
        s.lse = torch.empty(layers, B, c["q_heads"], device="cuda")
    s.params = [_params(c, t) for t in range(c["interval"])]
    s.graph = None
    if c["graph"]:
        _decode(s)                              # everything the first call sets up happens outside the capture
        torch.cuda.synchronize()
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            _decode(s)
    return s


def _params(c, t):
    if c["kind"] == "dense":
        return tb.select_params(-1)
    return tb.select_params(c["budget"], c["sinks"], c["recent"], c["radius"], NMODES[c["nmode"]], c["interval"], t,
                            REDUCES[c["reduce"]])


def _decode(s):
    """`interval` decode steps over the cached tokens."""
    c, B = s.c, s.c["batch"]
    for t, p in enumerate(s.params):
        for (l0, n) in _groups(c):
            if c["kind"] == "step":
                keep = s.idx is not None and t == 0
                s.ctx.select_topk(l0, n, None, B, s.q_imp[l0:l0 + n], p, s.idx[l0:l0 + n] if keep else None,
                                  s.cnt[l0:l0 + n] if keep else None)
            for l in range(l0, l0 + n):
                s.ctx.sparse_decode_attention(l, 1, None, B, s.q[t, l], p, s.out[t, l], lse=None if s.lse is None else s.lse[l])


def _prefill(s):
    for b in range(s.c["batch"]):
        s.ctx.reset_sequence(b)
    for l in range(s.c["layers"]):
        s.ctx.append_kv(l, 1, None, s.lengths, s.k[l], s.v[l])
    s.ctx.project_keys(0, s.c["layers"], None, s.zeros, s.lengths)


def _request(s):
    c, ctx, B = s.c, s.ctx, s.c["batch"]
    _prefill(s)
    done = s.lengths                            # projected tokens per sequence
    for t, p in enumerate(s.params):
        now = [L + t + 1 for L in s.lengths]
        refresh, r = t % c["interval"] == 0, t // c["interval"]
        for gi, (l0, n) in enumerate(_groups(c)):
            for l in range(l0, l0 + n):
                ctx.append_kv(l, 1, None, s.ones, s.k_new[t, l], s.v_new[t, l])
            if refresh:                         # the tokens since the last refresh, in one batch
                ctx.project_keys(l0, n, None, done, now)
                status = tb.predict_importance_queries(s.hidden[r, gi], scratch=s.scratch, q_imp=s.q_imp[r, gi], **s.predictors[gi])
                if status != tb.TB_OK:
                    raise tb.TBError(status, "predict_importance_queries")
            ctx.select_topk(l0, n, None, B, s.q_imp[r, gi], p, s.idx[r, l0:l0 + n] if refresh else None,
                            s.cnt[r, l0:l0 + n] if refresh else None)
            for l in range(l0, l0 + n):
                ctx.sparse_decode_attention(l, 1, None, B, s.q[t, l], p, s.out[t, l])
        if refresh:
            done = now


def run(state):
    s = state
    kind = s.c["kind"]
    if kind == "predict":
        for i, p in enumerate(s.predictors):
            status = tb.predict_importance_queries(s.hidden[i], scratch=s.scratch, q_imp=s.q_imp[i], **p)
            if status != tb.TB_OK:
                raise tb.TBError(status, "predict_importance_queries")
        return s.q_imp
    if kind == "prefill":
        _prefill(s)
        return s.out
    if kind == "request":
        _request(s)
        return {"out": s.out, "idx": s.idx, "cnt": s.cnt, "kimp": s.kimp}
    if s.graph is not None:
        s.graph.replay()
    else:
        _decode(s)
    return {"out": s.out, "lse": s.lse, "idx": s.idx, "cnt": s.cnt}
