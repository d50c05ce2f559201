"""The work a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values; its "op" says which public entry points one pass goes through:

  layers   ``LayerPath``: a prompt's observed layers, every step of the method (scoring, pooling, rank statistic,
           per-head top-k, K/V compaction), issued call by call or replayed from a captured CUDA graph
  score    ``asl_score_layer`` (two passes over K) or ``asl_score_layer_lse`` (the caller's attention has kept the
           window rows' log-sum-exp) on its own
  rank     ``asl_rank_stat`` on a full ring of rank rows
  select   ``asl_select_topk`` and ``asl_compact_kv`` on given scores: per-layer compression without layer selection
  oneshot  ``asl_select_topk`` on the aggregate (one head) and ``asl_compact_rows``: the selection layer's hidden states
  static   ``asl_rank_desc_static``: a rank row without context, workspace or allocation

A rank row, and a kept list whose boundary falls among near-equal scores, are discontinuous functions of the scores:
two correct scorers that round differently order such tokens differently.  So the tail's whole-number outputs are
compared where the scores are given ("rank", "select", "oneshot", "static": exactly), the scores where no selection
follows ("score"), and in "layers" the window attends to planted passages that fill the budget, halo of the pooling
included, so that the kept sets do not hang on rounding; there the rank rows show through the statistic they give.
"""
import math
import random

import numpy as np
import torch

from paper_2601_07667_b200 import binding as B

D = 128                                       # head dimension of every configuration
HEADS = ((8, 2), (32, 8), (28, 4), (64, 8))   # query heads / kv heads of the repository's configurations and tests
TAU = 0.3


def _layers(name, heads, window, tokens, keep, layers, requests=1, pool=7, pool_mode="avg", keys="bf16", issue="calls",
            free_sms=0, tails=1, latch=False):
    c = {"op": "layers", "q_heads": heads[0], "kv_heads": heads[1], "window": window, "tokens": tokens, "keep": keep,
         "layers": layers, "requests": requests, "pool": pool, "pool_mode": pool_mode, "keys": keys, "issue": issue,
         "free_sms": free_sms, "tails": tails, "latch": latch}
    return dict(c, name=name) if name else c


def _score(name, heads, window, tokens, requests=1, pool=7, pool_mode="avg", lse=False):
    c = {"op": "score", "q_heads": heads[0], "kv_heads": heads[1], "window": window, "tokens": tokens,
         "requests": requests, "pool": pool, "pool_mode": pool_mode, "lse": lse}
    return dict(c, name=name) if name else c


def _rank(name, tokens, requests, rows):
    c = {"op": "rank", "tokens": tokens, "requests": requests, "rows": rows, "window": 32, "keep": 0.1}
    return dict(c, name=name) if name else c


def _select(name, heads, tokens, requests, keep):
    c = {"op": "select", "q_heads": heads[0], "kv_heads": heads[1], "tokens": tokens, "requests": requests, "keep": keep,
         "window": 32}
    return dict(c, name=name) if name else c


def _oneshot(name, tokens, requests, keep, row_bytes):
    c = {"op": "oneshot", "tokens": tokens, "requests": requests, "keep": keep, "row_bytes": row_bytes, "window": 64}
    return dict(c, name=name) if name else c


def _static(name, tokens):
    c = {"op": "static", "tokens": tokens}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call there is: one request's rank row in a host that may not allocate
        _static("rank_row_static_4k", 4096),
        # the tiny four-layer stack: a short prompt on a small model, where launches and latency count
        _layers("layers_small_4k", (8, 2), 32, 4096, 0.125, 4),
        # the 8B-shaped layer sweep at 32K tokens: a full ring's worth of layers, the library's default launch settings
        _layers("layers_8b_32k", (32, 8), 64, 32768, 0.0625, 8),
        # the long-context request as the benchmark issues it: spare SMs, two side streams, one CUDA graph
        _layers("layers_8b_128k_graph", (32, 8), 64, 131072, 0.03125, 4, issue="graph", free_sms=16, tails=2),
        # ragged batched prefill, eight requests of 8K to 64K tokens, 10 % budgets, the controller on the device
        _layers("layers_8b_ragged", (32, 8), 32, 65536, 0.1, 2, requests=8, free_sms=16, tails=2, latch=True),
        # wide groups, 128 window rows and max pooling: twice the contraction per key of any other case
        _layers("layers_wide_max_64k", (64, 8), 128, 65536, 0.0625, 2, pool=5, pool_mode="max"),
        # a quantised (E4M3) key cache on the seven-queries-per-head layout, an odd length
        _layers("layers_7b_fp8_48k", (28, 4), 64, 49999, 0.05, 3, keys="fp8", free_sms=16, tails=2),
        # one pass over K: the caller's fused attention has the log-sum-exp of the window rows
        _score("score_lse_128k", (32, 8), 64, 131072, lse=True),
        # an observation window that is not a multiple of 32, on a ragged pair of prompts
        _score("score_window24_16k", (32, 8), 24, 16384, requests=2, pool=5),
        # the rank statistic alone over eight layers' rows, an odd number of tokens
        _rank("rank_stat_100k", 100003, 1, 8),
        # per-head compression that keeps half of every prompt: budgets that are a large part of the context
        _select("select_half_24k", (32, 8), 24001, 4, 0.5),
        # the selection layer: one list on the aggregate, then rows of hidden states (4096 bf16 channels)
        _oneshot("oneshot_hidden_96k", 98304, 1, 0.04, 8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_one(rng):
    op = rng.choice(("layers",) * 5 + ("score",) * 3 + ("rank", "select", "oneshot", "static"))
    if op == "layers":
        heads, window = rng.choice(HEADS), rng.choice((32, 64, 128))
        pool_mode = rng.choice(("avg", "avg", "avg", "max"))
        keys = rng.choice(("bf16", "bf16", "bf16", "fp8")) if pool_mode == "avg" else "bf16"
        return _layers(None, heads, window, _log_int(rng, 1500, 131072), round(math.exp(rng.uniform(math.log(0.02), math.log(0.25))), 4),
                       rng.randint(1, 8), rng.choice((1, 1, 2, 3, 8)), rng.choice((5, 7)), pool_mode, keys,
                       rng.choice(("calls", "calls", "graph")), *rng.choice(((0, 1), (16, 2))), rng.random() < 0.25)
    if op == "score":
        lse = rng.random() < 0.4
        window = rng.choice((32, 64, 128) if lse else (8, 16, 20, 24, 40, 48, 64, 100))
        return _score(None, rng.choice(HEADS), window, _log_int(rng, 1500, 131072 if lse else 32768), rng.choice((1, 1, 2, 4)),
                      rng.choice((3, 5, 7)), rng.choice(("avg", "avg", "max")), lse)
    if op == "rank":
        return _rank(None, _log_int(rng, 2000, 260000), rng.choice((1, 1, 2, 8)), rng.choice((2, 4, 8)))
    if op == "select":
        return _select(None, rng.choice(HEADS), _log_int(rng, 1500, 131072), rng.choice((1, 2, 4)), round(math.exp(rng.uniform(math.log(0.02), math.log(0.6))), 4))
    if op == "oneshot":
        return _oneshot(None, _log_int(rng, 2000, 131072), rng.choice((1, 2, 4)), round(math.exp(rng.uniform(math.log(0.02), math.log(0.3))), 4),
                        rng.choice((2048, 7168, 8192)))
    return _static(None, _log_int(rng, 300, 262144))


def draw(rng):
    """One more case of the ranges the listed ones stand for, no larger than the largest of them."""
    cost = lambda c: (lambda w: max(w["bytes"], w["flops"] / 50.0))(work(c))  # noqa: E731
    most = max(cost(c) for c in listed())
    while True:
        c = _draw_one(rng)
        if cost(c) <= most:
            return c


# ---- shapes ---------------------------------------------------------------------------------------
def _lengths(c):
    """Tokens of every request; a batch is ragged: lengths spread from an eighth of "tokens" up to it."""
    n, b = c["tokens"], c["requests"]
    if b == 1:
        return [n]
    r = random.Random(n * 31 + b)
    low = max(n // 8, 3 * c["window"] + 64)
    return [max(low, r.randint(low, max(low, n))) for _ in range(b)]


def _budgets(c):
    return [min(n, max(int(n * c["keep"]), c["window"] + 48)) for n in _lengths(c)]


def work(case):
    """Bytes and operations of one pass: K and Q once, V only where rows are kept, every output once; one Q.K^T."""
    op = case["op"]
    if op == "static":
        return {"bytes": 8 * case["tokens"], "flops": 0}
    n, kept = sum(_lengths(case)), sum(_budgets(case)) if "keep" in case else 0
    T = n - case["requests"] * case["window"]
    if op == "rank":      # scores, the earlier rows, the new row
        return {"bytes": 4 * T * (1 + case["rows"]) + 64 * case["requests"], "flops": 0}
    if op == "oneshot":   # scores, list, rows in and out
        return {"bytes": 4 * T + 4 * kept + 2 * kept * case["row_bytes"], "flops": 0}
    Hk = case["kv_heads"]
    if op == "select":    # scores, lists, K and V rows in and out
        return {"bytes": Hk * (4 * T + 4 * kept + 8 * kept * D), "flops": 0}
    Hq, W = case["q_heads"], case["window"]
    kb = 1 if case.get("keys") == "fp8" else 2
    bytes_ = kb * n * Hk * D + 2 * case["requests"] * Hq * W * D + 4 * (Hk + 1) * T
    flops = 2 * n * Hq * W * D
    if op == "score":
        return {"bytes": bytes_ + (4 * case["requests"] * Hq * W if case["lse"] else 0), "flops": flops}
    bytes_ += 4 * T + kept * Hk * (4 + kb * D + 4 * D)          # the rank row; lists, K rows out, V rows in and out
    return {"bytes": case["layers"] * bytes_, "flops": case["layers"] * flops}


def tolerance(case):
    """Scores are fp32 sums of fp32 exponentials of bf16 contractions: a logit's rounding (about 1e-5) and a short
    exponential (about 1e-4 in a term, of either sign) are what another scorer may differ by.  Everything whose
    inputs are given scores is integers and copied rows."""
    if case["op"] in ("layers", "score"):
        return {"rel": 1e-4, "max": 2e-3}
    return "exact"


# ---- inputs ---------------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape, dtype=torch.float32):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _directions(g, c):
    u = _randn(g, c["requests"], c["kv_heads"], D)
    return u / u.norm(dim=-1, keepdim=True)


def _queries(g, c, u):
    """Window queries [B][H_q][W][d] that lean towards their kv head's direction (cosine one half)."""
    lean = (math.sqrt(D / 3.0) * u).repeat_interleave(c["q_heads"] // c["kv_heads"], dim=1)
    return (_randn(g, c["requests"], c["q_heads"], c["window"], D) + lean[:, :, None]).to(torch.bfloat16)


def _passages(c, seed):
    """Per kv head, packed positions of the tokens of planted passages.  With the pooling's halo the passages of a
    request take exactly its budget of past tokens; each lies somewhere in a slot of its own."""
    rng, r, W, H = np.random.default_rng([int(seed), 77]), c["pool"] // 2, c["window"], c["kv_heads"]
    out, start = [], 0
    for n, budget in zip(_lengths(c), _budgets(c)):
        T, k = n - W, budget - W
        P = max(1, min(32, k // (2 * r + 16)))
        lens = np.array([k // P + (i < k % P) - 2 * r for i in range(P)])
        slot = T // P
        for h in range(H):
            first = np.arange(P) * slot + r + (rng.random(P) * (slot - 2 * r - lens + 1)).astype(np.int64)
            tok = np.concatenate([np.arange(f, f + m) for f, m in zip(first, lens)])
            out.append((start + tok) * H + h)
        start += n
    return torch.from_numpy(np.concatenate(out)).cuda()


def _keys(g, c, u, planted, strength):
    """K [tokens][H_k][d] bf16: Gaussian background, planted rows along the direction with noise of their own."""
    n, H = sum(_lengths(c)), c["kv_heads"]
    k = _randn(g, n, H, D, dtype=torch.bfloat16)
    request = torch.repeat_interleave(torch.arange(c["requests"]), torch.tensor(_lengths(c))).cuda()
    rows = k.view(n * H, D)
    rows[planted] = (0.75 * rows[planted].float() + strength * math.sqrt(D) * u[request[planted // H], planted % H]).to(torch.bfloat16)
    return k


def _path(c, k_scale=None):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    free = c.get("free_sms", 0)
    rows = c.get("layers", c.get("rows", 2))
    return B.LayerPath(n_q_heads=c.get("q_heads", 1), n_kv_heads=c.get("kv_heads", 1), head_dim=D, window=c["window"],
                       pool_kernel=c.get("pool", 7), pool_mode=B.ASL_POOL_MAX if c.get("pool_mode") == "max" else B.ASL_POOL_AVG,
                       seqlens=_lengths(c), budgets=_budgets(c) if "keep" in c else _lengths(c), l_min=1,
                       l_obs=max(2, min(8, rows)), tau=TAU, score_ctas=sms - free if free else 0, tail_streams=c.get("tails", 1),
                       k_dtype=B.ASL_K_FP8_E4M3 if k_scale else B.ASL_K_BF16, k_scale=k_scale)


def _pooled_scores(g, rows, T, scale=1.0):
    """Score rows as pooled attention gives them: positive, heavy tailed, smooth over a few neighbours."""
    x = torch.exp(scale * _randn(g, rows, T) - 9.0)
    return torch.nn.functional.avg_pool1d(x[:, None], 7, 1, 3)[:, 0].contiguous()


def _window_lse(q, k, c):
    """log-sum-exp of every window row over the keys it sees, [B][H_q][W], as a fused attention forward keeps it."""
    W, G = c["window"], c["q_heads"] // c["kv_heads"]
    out = torch.empty((c["requests"], c["q_heads"], W), dtype=torch.float32, device="cuda")
    hidden = torch.ones(W, W, device="cuda", dtype=torch.bool).triu(1)
    start = 0
    for b, n in enumerate(_lengths(c)):
        for h in range(c["kv_heads"]):
            s = q[b, h * G:(h + 1) * G].reshape(G * W, D).float() @ k[start:start + n, h].float().T / math.sqrt(D)
            s = s.view(G, W, n)
            s[:, :, n - W:].masked_fill_(hidden, float("-inf"))
            out[b, h * G:(h + 1) * G] = torch.logsumexp(s, dim=-1)
        start += n
    return out


def prepare(case, seed):
    g, c = _generator(seed), case
    op = c["op"]
    if op == "static":
        scores = _pooled_scores(g, 1, c["tokens"])[0]
        return {"op": op, "scores": scores, "rank": torch.empty(c["tokens"], dtype=torch.int32, device="cuda")}
    if op == "layers":
        u, planted = _directions(g, c), _passages(c, seed)
        steps = []
        for _ in range(c["layers"]):
            k = _keys(g, c, u, planted, 1.25)
            steps.append([_queries(g, c, u), k, _randn(g, *k.shape, dtype=torch.bfloat16)])
        scale = None
        if c["keys"] == "fp8":                  # one scale per kv head of the plan
            scale = torch.stack([s[1].abs().amax(dim=(0, 2)) for s in steps]).amax(dim=0).float() / 448.0
            for s in steps:
                s[1] = (s[1].float() / scale[None, :, None]).to(torch.float8_e4m3fn).view(torch.uint8)
            scale = scale.tolist()
        path = _path(c, scale)
        if c["latch"]:
            path.set_controller(B.ASL_CONTROLLER_LATCH)
        state = {"op": op, "path": path, "steps": steps, "graph": None}
        if c["issue"] == "graph":
            run(state)                          # once by calls, as capturing asks for
            path.reset()
            state["graph"] = path.capture([(*s, l) for l, s in enumerate(steps)])
        return state
    path = _path(c)
    state = {"op": op, "path": path}
    T = path.sum_T
    if op == "score":
        u = _directions(g, c)
        few = torch.from_numpy(np.random.default_rng(int(seed)).integers(0, path.sum_tokens * c["kv_heads"], 8 * c["kv_heads"])).cuda()
        state["q"], state["k"] = _queries(g, c, u), _keys(g, c, u, few, 1.0)
        state["lse"] = _window_lse(state["q"], state["k"], c) if c["lse"] else None
        state["kv"], state["agg"] = torch.empty((c["kv_heads"], T), device="cuda"), torch.empty(T, device="cuda")
    elif op == "rank":
        # the earlier layers' rows are in the ring: scores that share a per-token salience from layer to layer
        lasting = _pooled_scores(g, 1, T)[0]
        state["layer"] = c["rows"] - 1
        for layer in range(c["rows"]):
            state["agg"] = lasting * _pooled_scores(g, 1, T, 0.5)[0]
            B.asl_rank_stat(path.ctx, state["agg"], layer, layer + 1, path.rank_ring, path.stat, path.workspace, path.ws_bytes)
            torch.cuda.current_stream().synchronize()          # the scores are replaced by the next layer's
    elif op == "select":
        state["kv"] = _pooled_scores(g, c["kv_heads"], T)
        state["k"] = _randn(g, path.sum_tokens, c["kv_heads"], D, dtype=torch.bfloat16)
        state["v"] = _randn(g, path.sum_tokens, c["kv_heads"], D, dtype=torch.bfloat16)
    else:
        state["agg"] = _pooled_scores(g, 1, T)[0]
        state["x"] = _randn(g, path.sum_tokens, c["row_bytes"] // 2, dtype=torch.bfloat16)
        state["idx"] = torch.empty(path.sum_kept, dtype=torch.int32, device="cuda")
        state["out"] = torch.empty((path.sum_kept, c["row_bytes"] // 2), dtype=torch.bfloat16, device="cuda")
        state["row_bytes"] = c["row_bytes"]
    return state


def run(state):
    op = state["op"]
    if op == "static":
        B.asl_rank_desc_static(state["scores"], state["scores"].numel(), state["rank"])
        return {"rank": state["rank"]}
    p = state["path"]
    if op == "layers":
        p.reset()                               # a new prompt
        if state["graph"] is not None:
            state["graph"].replay()
        else:
            for layer, (q, k, v) in enumerate(state["steps"]):
                p.run_layer(q, k, v, layer)
            p.join()
        # the statistic as a caller reads it: var_top, init_var and rel of every request
        return {"scores_kv": p.scores_kv, "scores_agg": p.scores_agg, "idx": p.idx, "k_out": p.k_out, "v_out": p.v_out,
                "stat": p.stat.view(torch.float64)[:, 5:8]}
    if op == "score":
        if state["lse"] is None:
            B.asl_score_layer(p.ctx, state["q"], state["k"], state["kv"], state["agg"], p.workspace, p.ws_bytes)
        else:
            B.asl_score_layer_lse(p.ctx, state["q"], state["k"], state["lse"], state["kv"], state["agg"], p.workspace, p.ws_bytes)
        return {"scores_kv": state["kv"], "scores_agg": state["agg"]}
    if op == "rank":
        layer = state["layer"]
        B.asl_rank_stat(p.ctx, state["agg"], layer, min(layer + 1, p.l_obs), p.rank_ring, p.stat, p.workspace, p.ws_bytes)
        return {"ring": p.rank_ring, "stat": p.stat}
    if op == "select":
        B.asl_select_topk(p.ctx, state["kv"], p.H_k, p.idx, p.workspace, p.ws_bytes)
        B.asl_compact_kv(p.ctx, state["k"], state["v"], p.idx, p.k_out, p.v_out)
        return {"idx": p.idx, "k_out": p.k_out, "v_out": p.v_out}
    B.asl_select_topk(p.ctx, state["agg"], 1, state["idx"], p.workspace, p.ws_bytes)
    B.asl_compact_rows(p.ctx, state["x"], state["idx"], state["out"], state["row_bytes"])
    return {"idx": state["idx"], "rows": state["out"]}
