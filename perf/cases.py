"""What this framework is asked to do, as cases that can be timed: decode steps of a budgeted KV
cache from one tiny sequence to large batches, the options such a cache is run with, a chat turn's
chunk and its compression, attention without a handle, and the training-side sampler.

The inputs follow the recipe of the package's synthetic workloads: N(0, 1) keys and values, four
sink tokens with keys x 4, 1% heavy hitters whose keys are 4 u + N(0, 1) for a per-row direction u,
queries 0.1 u + N(0, 1), all bfloat16. Policy weights follow PyTorch's rule for linear layers.

A decode-step state is a cache in its steady state: budget - W prompt tokens and W = 64 decode steps
(the entropy window; fewer on the smallest budgets) fill it to the budget, and run() takes the next
step, which appends one token to every row, attends, scores and evicts one token from every row.
"""

import math

import numpy as np
import torch

from paper_2608_08878_gb300 import dc

WINDOW = 64   # w of the entropy feature (the library's default)
POOL = 72     # different step inputs a state holds, taken in turn


def _step(name, layers, batch, kvh, group, d, budget, scorer="policy", **kw):
    return dict(name=name, kind="step", layers=layers, batch=batch, kvh=kvh, group=group, d=d, budget=budget,
                scorer=scorer, hidden=kw.get("hidden", 128), layernorm=kw.get("layernorm", True))


def listed():
    return [
        # the smallest call: one layer, 2 KV heads of 64 dims, 128 tokens kept, a 64-wide policy
        # without LayerNorm (a unit of work that is all latency and launches)
        _step("step_tiny", 1, 1, 2, 2, 64, 128, hidden=64, layernorm=False),
        # one Mistral-7B layer of one sequence, 8K context at 25%: a model that calls the cache
        # layer by layer
        _step("step_1layer_seq1", 1, 1, 8, 4, 128, 2048),
        # all 32 layers of one sequence, 4K context at 10%: interactive decoding
        _step("step_seq1_ctx4k_10", 32, 1, 8, 4, 128, 410),
        # one sequence with a long memory: 32K context at 50%
        _step("step_seq1_ctx32k_50", 32, 1, 8, 4, 128, 16384),
        # the benchmark: 8 sequences, 32K context at 25%
        _step("step_seq8_ctx32k_25", 32, 8, 8, 4, 128, 8192),
        # a large serving batch of short contexts: 64 sequences, 4K at 10%
        _step("step_seq64_ctx4k_10", 32, 64, 8, 4, 128, 410),
        # the same benchmark with eight query heads per KV head (70B-class models: 4 KV heads)
        _step("step_gqa8_seq8_ctx32k_25", 32, 8, 4, 8, 128, 8192),
        # the head-level hybrid: a fifth of the heads keep their full 16K context, the others share
        # the rest of a 25% budget; two sequences
        dict(name="step_hybrid_seq2_ctx16k", kind="hybrid", layers=32, batch=2, kvh=8, group=4, d=128,
             context=16384),
        # a caller that wants the scores: decode step, scores read back, eviction as a call of its own
        dict(name="decode_scores_evict_seq1", kind="scores", layers=32, batch=1, kvh=8, group=4, d=128,
             budget=1638),
        # a chat turn, or a chunk of a prompt: 24576 tokens appended to a cache at its budget, whose
        # first decode step compresses 32769 tokens back to 8192
        dict(name="turn_24k_compress_8k", kind="turn", layers=8, batch=4, kvh=8, group=4, d=128,
             budget=8192, chunk=24576),
        # attention over caller-owned buffers with no handle and no allocation: one Mistral-7B layer,
        # 8 sequences of 8K tokens
        dict(name="attend_noalloc_seq8_8k", kind="attend", rows=64, n=8192, group=4, d=128),
        # the training side: 64 sampled subsets of 1024 of 4096 tokens, with their log-probabilities
        dict(name="gumbel_top_b_64x4096", kind="gumbel", rows=64, length=4096, budget=1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges, no dearer than the benchmark."""
    kind = rng.choices(["step", "hybrid", "scores", "turn", "attend", "gumbel"], [60, 6, 8, 6, 10, 10])[0]
    if kind == "attend":
        while True:
            c = dict(kind=kind, rows=_log(rng, 1, 256), n=_log(rng, 64, 32768), group=rng.choice([1, 2, 4, 4, 8]),
                     d=rng.choice([64, 128, 128]))
            if 1 << 16 <= c["rows"] * c["n"] * c["d"] <= 1 << 29:
                return c
    if kind == "gumbel":
        while True:
            c = dict(kind=kind, rows=_log(rng, 1, 256), length=_log(rng, 128, 8192))
            c["budget"] = max(1, int(c["length"] * rng.uniform(0.05, 0.5)))
            if c["rows"] * c["length"] * c["budget"] <= 1 << 30:
                return c
    while True:
        c = dict(kind=kind, layers=rng.choice([1, 2, 4, 8, 16, 32, 32]), batch=_log(rng, 1, 64),
                 kvh=rng.choice([2, 4, 8, 8]), group=rng.choice([1, 2, 4, 4, 8]), d=rng.choice([64, 128, 128]))
        rows = c["layers"] * c["batch"] * c["kvh"]
        if kind == "hybrid":
            c["context"] = _log(rng, 1024, 16384)
            tokens = rows * c["context"]
        else:
            c["budget"] = _log(rng, 96, 16384)
            tokens = rows * (c["budget"] + 1)
        if kind == "step":
            c["scorer"] = rng.choice(["policy", "policy", "policy", "h2o", "streaming", "global"])
            c["hidden"], c["layernorm"] = rng.choice([(128, True), (128, True), (64, False)])
        if kind == "turn":
            c["chunk"] = _log(rng, 64, 24576)
            tokens += rows * c["chunk"]
        most = (1 << 24) if kind == "step" else (1 << 23)
        if 1 << 12 <= tokens <= most and rows <= 16384:
            return c


# ---------------------------------------------------------------------------
# Inputs: from the seed alone, on the GPU
# ---------------------------------------------------------------------------
def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(seed * 16 + stream)


def _rows(c):
    return c["layers"] * c["batch"] * c["kvh"]


def _directions(c, seed):
    return torch.randn((c["layers"], c["batch"], c["kvh"], c["d"]), device="cuda", generator=_gen(seed, 0))


def _tokens(c, seed, stream, T, sinks):
    """bf16 k, v [layers][batch][kvh][T][d] of T prompt tokens."""
    L, b, kvh, d = c["layers"], c["batch"], c["kvh"], c["d"]
    u, g = _directions(c, seed), _gen(seed, stream)
    k = torch.empty((L, b, kvh, T, d), dtype=torch.bfloat16, device="cuda")
    v = torch.empty_like(k)
    for layer in range(L):
        x = torch.randn((b, kvh, T, d), device="cuda", generator=g)
        if sinks:
            x[:, :, :4] *= 4.0
        hot = torch.rand((b, kvh, T, 1), device="cuda", generator=g) < 0.01
        if sinks:
            hot[:, :, :4] = False
        x += hot * (4.0 * u[layer])[:, :, None]
        k[layer] = x
        v[layer] = x.normal_(generator=g)
    return k, v


def _steps(c, seed, count):
    """count decode steps' inputs: bf16 q [count][layers][batch][q heads][d], k, v [count][layers][batch][kvh][d]."""
    L, b, kvh, G, d = c["layers"], c["batch"], c["kvh"], c["group"], c["d"]
    u, g = _directions(c, seed), _gen(seed, 2)
    q = torch.empty((count, L, b, kvh * G, d), dtype=torch.bfloat16, device="cuda")
    k = torch.empty((count, L, b, kvh, d), dtype=torch.bfloat16, device="cuda")
    v = torch.empty_like(k)
    for s in range(count):
        x = torch.randn((L, b, kvh, G, d), device="cuda", generator=g)
        q[s] = (x + 0.1 * u[:, :, :, None]).view(L, b, kvh * G, d)
        k[s] = torch.randn((L, b, kvh, d), device="cuda", generator=g)
        v[s] = torch.randn((L, b, kvh, d), device="cuda", generator=g)
    return q, k, v


def _policy(c, seed):
    """[W1 (H x 5) | b1 | gamma | beta | w2 | b2], the linear layers as PyTorch draws them."""
    H, r = c.get("hidden", 128), np.random.RandomState(seed % (1 << 31))
    lin = lambda n, fan: r.uniform(-1, 1, n) / math.sqrt(fan)  # noqa: E731
    return np.concatenate([lin(5 * H, 5), lin(H, 5), 1 + 0.1 * r.randn(H), 0.1 * r.randn(H), lin(H, H),
                           lin(1, H)]).astype(np.float32)


def _warm(c):
    return min(WINDOW, c["budget"] // 2)


def _cache(c, capacity, budget, **kw):
    return dc.DistillCache(c["layers"], c["kvh"], c["d"], capacity, budget, batch=c["batch"],
                           q_heads=c["kvh"] * c["group"], window=WINDOW, mlp_hidden=c.get("hidden", 128),
                           layernorm=int(c.get("layernorm", True)), **kw)


def _state(c, cache, seed):
    s = dict(kind=c["kind"], cache=cache, at=0)
    s["q"], s["k"], s["v"] = (x.unbind(0) for x in _steps(c, seed, POOL))
    s["out"] = torch.empty(s["q"][0].shape, dtype=torch.float32, device="cuda")
    return s


def _next(s):
    i = s["at"] % POOL
    s["at"] += 1
    return s["q"][i], s["k"][i], s["v"][i]


def prepare(case, seed):
    c = case
    if c["kind"] == "attend":
        g = _gen(seed, 0)
        shape = (c["rows"], c["n"], c["d"])
        k = torch.randn(shape, device="cuda", generator=g).bfloat16()
        v = torch.randn(shape, device="cuda", generator=g).bfloat16()
        q = torch.randn((c["rows"], c["group"], c["d"]), device="cuda", generator=g).bfloat16()
        return dict(kind="attend", q=q, kv=(k, v), out=torch.empty(q.shape, dtype=torch.float32, device="cuda"))
    if c["kind"] == "gumbel":
        g = _gen(seed, 0)
        scores = torch.randn((c["rows"], c["length"]), device="cuda", generator=g)
        noise = -torch.log(torch.empty_like(scores).exponential_(generator=g))
        return dict(kind="gumbel", scores=scores, noise=noise, budget=c["budget"])
    if c["kind"] == "hybrid":
        rows = _rows(c)
        cache = _cache(c, c["context"] + 1, max(1, c["context"] // 4))
        cache.set_policy(_policy(c, seed))
        cache.set_row_budgets(dc.head_level_hybrid_budgets(rows, c["context"], range(0, rows, 5), 0.25))
        cache.append(*_tokens(c, seed, 1, c["context"], True))
        s = _state(c, cache, seed)
        for _ in range(WINDOW):
            cache.step(*_next(s), out=s["out"])
        return s
    scorer = c.get("scorer", "policy")
    W = _warm(c)
    cache = _cache(c, c["budget"] + c.get("chunk", 0) + 1, c["budget"],
                   scorer={"h2o": 1, "streaming": 2}.get(scorer, 0), global_tokens=scorer == "global")
    cache.set_policy(_policy(c, seed))
    cache.append(*_tokens(c, seed, 1, c["budget"] - W, True))
    s = _state(c, cache, seed)
    for _ in range(W):
        cache.step(*_next(s), out=s["out"])
    if c["kind"] == "turn":
        s["chunk"] = _tokens(c, seed, 3, c["chunk"], False)
    return s


def run(state):
    s = state
    if s["kind"] in ("step", "hybrid"):
        return s["cache"].step(*_next(s), out=s["out"])
    if s["kind"] == "scores":
        out = s["cache"].decode_step(*_next(s), out=s["out"])
        scores = s["cache"].buffer(dc.BUF_SCORE)
        s["cache"].evict()
        return out, scores
    if s["kind"] == "turn":
        s["cache"].append(*s["chunk"])
        return s["cache"].step(*_next(s), out=s["out"])
    if s["kind"] == "attend":
        return dc.attend_noalloc(s["q"], *s["kv"], out=s["out"])
    return dc.gumbel_top_b(s["scores"], s["noise"], s["budget"])


def work(case):
    c = case
    if c["kind"] == "attend":
        return {"bytes": c["rows"] * (c["n"] * 4 * c["d"] + 6 * c["group"] * c["d"]),
                "flops": c["rows"] * c["n"] * 4 * c["group"] * c["d"]}
    if c["kind"] == "gumbel":
        # scores and noise in, indices and log-probabilities out; a logistic and a few products per token
        return {"bytes": c["rows"] * (8 * c["length"] + 4 * c["budget"] + 4), "flops": c["rows"] * c["length"] * 16}
    d, G, rows = c["d"], c["group"], _rows(c)
    if c["kind"] == "hybrid":
        b = dc.head_level_hybrid_budgets(rows, c["context"], range(0, rows, 5), 0.25)
        tokens = int(np.minimum(b, c["context"]).sum()) + rows
    else:
        tokens = rows * (c["budget"] + c.get("chunk", 0) + 1)
    # per token: K and V read, position read, window sums (S, Z as double-float pairs) read and
    # written, |v| left out (it follows from V); per row: the new pair and its state written, its
    # query read, the output written, one slot moved
    slot = 4 * d + 20
    h2o = 8 if c.get("scorer") == "h2o" else 0
    state = 4 if c.get("scorer") == "global" else 36
    byte = tokens * (4 * d + state + h2o) + rows * (3 * slot + 4 * d + 6 * G * d)
    if c["kind"] == "scores":
        byte += tokens * 4
    if c["kind"] == "turn":
        # the chunk read and written with its state; survivors past the budget moved into the holes
        n, B = c["budget"] + c["chunk"] + 1, c["budget"]
        byte += rows * (c["chunk"] * (8 * d + 20) + B * (n - B) // n * 2 * slot)
    # QK^T of the current, the previous and the departing queries, PV, the policy's two layers
    flops = tokens * (2 * d * G * 4 + 12 * c.get("hidden", 128))
    return {"bytes": byte, "flops": flops}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits
# ---------------------------------------------------------------------------
def _attend64(q, k, v):
    """q [r][G][d], k, v [r][n][d] in 64 bits -> the output and the weights' logits."""
    s = torch.einsum("rgd,rnd->rgn", q, k) / math.sqrt(q.shape[-1])
    return torch.einsum("rgn,rnd->rgd", torch.softmax(s, -1), v)


def _chunks(rows, n, d):
    step = max(1, (1 << 27) // (n * d))
    return [(r, min(rows, r + step)) for r in range(0, rows, step)]


def exact(case, seed):
    c = case
    if c["kind"] == "hybrid":
        return None  # which tokens the prompt compression kept hangs on near-ties of 32-bit scores
    if c["kind"] == "attend":
        s = prepare_inputs_attend(c, seed)
        return torch.cat([_attend64(*(x[a:b].double() for x in s)) for a, b in _chunks(c["rows"], c["n"], c["d"])])
    if c["kind"] == "gumbel":
        return None, _gumbel64(c, seed)
    rows, d, G, W = _rows(c), c["d"], c["group"], _warm(c)
    k0, v0 = (x.view(rows, -1, d) for x in _tokens(c, seed, 1, c["budget"] - W, True))
    q, kn, vn = _steps(c, seed, POOL)
    q = q[: W + 1].view(W + 1, rows, G, d)
    kn, vn = (x[: W + 1].view(W + 1, rows, d).transpose(0, 1) for x in (kn, vn))  # [rows][W + 1][d]
    ck, cv = (x.view(rows, -1, d) for x in _tokens(c, seed, 3, c["chunk"], False)) if c["kind"] == "turn" else (None, None)
    n = c["budget"] + c.get("chunk", 0) + 1
    outs, scores = [], []
    for a, b in _chunks(rows, n, d):
        parts_k, parts_v = [k0[a:b], kn[a:b, :W]], [v0[a:b], vn[a:b, :W]]
        if ck is not None:
            parts_k.append(ck[a:b])
            parts_v.append(cv[a:b])
        K = torch.cat(parts_k + [kn[a:b, W:]], 1).double()
        V = torch.cat(parts_v + [vn[a:b, W:]], 1).double()
        outs.append(_attend64(q[W, a:b].double(), K, V))
        if c["kind"] == "scores":
            scores.append(_scores64(c, seed, q[:, a:b].double(), K, V, W))
    out = torch.cat(outs).view(c["layers"], c["batch"], c["kvh"] * G, d)
    return (out, torch.cat(scores)) if c["kind"] == "scores" else out


def prepare_inputs_attend(c, seed):
    s = prepare(c, seed)
    return (s["q"],) + s["kv"]


def _scores64(c, seed, q, K, V, W):
    """Policy scores after the step: features over the window's queries, then the MLP."""
    n, d = K.shape[1], K.shape[2]
    Z = S = 0.0
    for s in range(max(0, W + 1 - WINDOW), W + 1):
        m = n - W + s  # tokens cached at step s
        p = torch.softmax(torch.einsum("rgd,rnd->rgn", q[s], K[:, :m]) / math.sqrt(d), -1)
        H = -torch.special.xlogy(p, p).sum(-1, keepdim=True)
        pad = torch.zeros((p.shape[0], n - m), dtype=p.dtype, device=p.device)
        Z = Z + torch.cat([p.sum(1), pad], 1)
        S = S + torch.cat([(p * H).sum(1), pad], 1)
    pos = torch.arange(n, device=K.device).double() / (n - 1)
    x = torch.stack([p.mean(1), V.norm(dim=-1), p.var(1, unbiased=False), S / Z, pos.expand_as(Z)], -1)
    w, H = torch.from_numpy(_policy(c, seed)).double().cuda(), c.get("hidden", 128)
    W1, b1, gam, bet, w2, b2 = w[: 5 * H].view(H, 5), *(w[(5 + i) * H: (6 + i) * H] for i in range(4)), w[9 * H]
    h = torch.nn.functional.layer_norm(x @ W1.T + b1, (H,), gam, bet, 1e-5)
    return torch.relu(h) @ w2 + b2


def _gumbel64(c, seed):
    """log P(a) = sum of the subset's scores - log e_B(exp(scores)), e_B by its recurrence in logarithms."""
    s = prepare(c, seed)
    x = s["scores"].double()
    idx = (s["scores"] + s["noise"]).topk(c["budget"], -1).indices
    e = torch.full((c["rows"], c["budget"] + 1), -math.inf, dtype=torch.float64, device="cuda")
    e[:, 0] = 0.0
    for i in range(c["length"]):
        e[:, 1:] = torch.logaddexp(e[:, 1:], e[:, :-1] + x[:, i: i + 1])
    return x.gather(1, idx).sum(1) - e[:, -1]
