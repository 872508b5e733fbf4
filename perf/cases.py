"""The work this framework is used for, as cases whose time and outputs can be measured.

Five kinds of pass, each through the public entry points a program calls:

- ``step``: one decode step of one attention layer, ``KVpopCache.step`` (delayed scorer,
  keep-or-drop, scatter, attention over the compressed cache).
- ``stack``: one decode step of several layers with their projections, ``DecodeStack``
  captured into a CUDA graph once and replayed, as a serving loop does.
- ``prompt``: one prompt batch through ``KVpopCache.prefill_attend`` (scores, compression,
  ranks, cutoffs, masked attention); or, with the mLSTM scorer, ``KVpopCache.prefill`` and
  the first generated token.
- ``train``: the scorer's training forward: ``topk_cutoff``, ``prompt_attention`` under the
  running top-k mask and ``future_target`` with its normalisers.
- ``target``: the exact training target: ``causal_lse`` and ``future_target``.

Prompt and decode tokens are N(0, 1) with a few outlier key channels, as in this
repository's workloads; every value follows from the seed alone.
"""
from __future__ import annotations

import math

import torch

from paper_2607_05061_gb300 import kvpop
from paper_2607_05061_gb300.stack import DecodeStack

RING = 16                # decode inputs a state holds; a step takes the next of them
GROUP = 4                # sequences whose prompt tensors are made at a time


def _case(kind, name=None, **kw):
    c = {"kind": kind, "batch": 1, "kv_heads": 8, "q_per_kv": 4, "head_dim": 128, "dtype": "bf16",
         "lo": 4096, "hi": 4096, "budget": 3072, "window": 16, "sinks": 0, "scorer_hidden": 256,
         "scorer": "gelu", "layers": 1, "hidden": 0, "log_gamma": 0.0, "lookahead": 0,
         "agg": "max"}
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: the fp32 layer of the `tiny` configuration, where latency counts
        _case("step", "step_tiny_fp32", batch=1, kv_heads=2, q_per_kv=2, head_dim=64, dtype="f32",
              lo=128, hi=128, budget=64, window=4, scorer_hidden=32),
        # the headline layer: 8x compression, batch 64 (the prompt is shorter than the
        # workload's 32768 tokens: a step reads the 4096 kept slots either way)
        _case("step", "step_cr8x", batch=64, lo=8192, hi=8192, budget=4096),
        # the same batch under the stateful mLSTM scorer, its budget just filled
        _case("step", "step_mlstm", batch=64, lo=4128, hi=4128, budget=4096, window=32,
              scorer="mlstm"),
        # one chat user: batch 1, the latency of a token through a few layers
        _case("stack", "stack_b1", batch=1, lo=4096, hi=4096, budget=3072, layers=4, hidden=4096),
        # a small serving batch at the 75% operating point (Qwen3-4B-shaped layers)
        _case("stack", "stack_b8", batch=8, lo=4096, hi=4096, budget=3072, layers=4, hidden=4096),
        # a large serving batch (two layers of the Qwen3-8B-shaped stack)
        _case("stack", "stack_b32", batch=32, lo=9000, hi=9000, budget=8192, layers=2, hidden=4096),
        # one long prompt at the 8x operating point
        _case("prompt", "prompt_32k", batch=1, lo=32768, hi=32768, budget=4096),
        # a ragged batch of ordinary prompts with sinks and decay, odd lengths
        _case("prompt", "prompt_ragged", batch=6, lo=233, hi=2801, budget=1024, window=32, sinks=4,
              log_gamma=-0.001),
        # prompts within the budget for a long generation, stateful scorer, first token
        _case("prompt", "prompt_mlstm", batch=8, lo=2011, hi=4009, budget=4096, window=32,
              scorer="mlstm"),
        # training forward of one layer: masked attention and the sparse target
        _case("train", "train_8k", batch=2, lo=8192, hi=8192, budget=1028, window=256, sinks=4),
        # the same in fp32 for a small d = 64 model, odd length
        _case("train", "train_fp32", batch=2, kv_heads=4, q_per_kv=2, head_dim=64, dtype="f32",
              lo=2039, hi=2039, budget=260, window=64, sinks=4, agg="mean"),
        # the exact target (dense normalisers) of longer training sequences
        _case("target", "target_16k", batch=1, lo=16384, hi=16384, window=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step_mlstm", "stack", "stack", "prompt", "prompt_mlstm", "train",
                       "train_fp32", "target"])
    if kind == "step":
        if rng.random() < 0.5:                      # small fp32 layers
            budget = _log(rng, 32, 1024)
            P = budget + _log(rng, 16, 1024)
            return _case("step", batch=_log(rng, 1, 4), kv_heads=rng.choice([2, 4]),
                         q_per_kv=rng.choice([1, 2, 4]), head_dim=64, dtype="f32", lo=P, hi=P,
                         budget=budget, window=rng.choice([4, 8, 16]),
                         scorer_hidden=rng.choice([32, 64, 128]))
        budget = _log(rng, 3072, 4096)              # large bf16 batches
        return _case("step", batch=rng.randint(56, 64), lo=budget + 64, hi=budget + _log(rng, 512, 4096),
                     budget=budget, sinks=rng.choice([0, 4]))
    if kind == "step_mlstm":
        budget, window = _log(rng, 3072, 4096), rng.choice([16, 32])
        return _case("step", batch=rng.randint(48, 64), lo=budget + window, hi=budget + window,
                     budget=budget, window=window, scorer="mlstm")
    if kind == "stack":
        batch, budget = _log(rng, 1, 32), _log(rng, 768, 8192)
        P = budget + _log(rng, 64, 1024)
        return _case("stack", batch=batch, lo=P, hi=P, budget=budget, layers=rng.choice([1, 2]),
                     hidden=rng.choice([2048, 2560, 4096]))
    if kind == "prompt":
        hi = _log(rng, 700, 16384)
        batch = max(1, min(8, 24576 // hi))
        budget = max(128, _log(rng, max(130, hi // 16), max(131, hi // 3)))
        return _case("prompt", batch=batch, lo=max(1, hi // rng.choice([1, 2, 8])), hi=hi,
                     budget=budget, window=rng.choice([16, 32]), sinks=rng.choice([0, 4]),
                     log_gamma=rng.choice([0.0, -0.001]))
    if kind == "prompt_mlstm":
        hi = _log(rng, 500, 4096)
        return _case("prompt", batch=_log(rng, 1, 8), lo=max(1, hi // 2), hi=hi, budget=4096,
                     window=rng.choice([16, 32]), scorer="mlstm")
    if kind == "train_fp32":
        S = _log(rng, 300, 2048)
        return _case("train", batch=_log(rng, 1, 2), kv_heads=rng.choice([2, 4]), q_per_kv=2,
                     head_dim=64, dtype="f32", lo=S, hi=S, budget=max(20, S // 8) + 4,
                     window=rng.choice([16, 64]), sinks=4, agg=rng.choice(["max", "mean"]))
    if kind == "train":
        S = _log(rng, 900, 8192)
        return _case("train", batch=_log(rng, 1, max(2, min(8, 16384 // S))), lo=S, hi=S,
                     budget=max(64, S // 8) + 4, window=rng.choice([64, 256]), sinks=4,
                     agg=rng.choice(["max", "mean"]))
    S = _log(rng, 1500, 16384)
    return _case("target", batch=max(1, min(4, 16384 // S)), lo=S, hi=S,
                 window=rng.choice([64, 256]), lookahead=rng.choice([0, 0, 1024]),
                 agg=rng.choice(["max", "mean"]))


# ---------------------------------------------------------------------- inputs from the seed
def _gen(seed, tag, device):
    g = torch.Generator(device=device)
    g.manual_seed((seed * 1000003 + tag * 7919 + 17) % (1 << 62))
    return g


def _randn(shape, seed, tag, dtype=torch.float32, scale=1.0, device="cuda"):
    t = torch.randn(shape, generator=_gen(seed, tag, device), dtype=torch.float32, device=device)
    return (t.mul_(scale) if scale != 1.0 else t).to(dtype)


def _dtype(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _lengths(c, seed):
    """Prompt lengths: uniform in [lo, hi], the last one hi."""
    g = torch.Generator()
    g.manual_seed(seed * 31 + 7)
    L = torch.randint(c["lo"], c["hi"] + 1, (c["batch"],), generator=g).tolist()
    return L[:-1] + [c["hi"]]


def _key_scale(c):
    """Outlier key channels: 4 of the channels of d = 128 heads, ten times the others."""
    s = torch.ones(c["head_dim"], device="cuda")
    if c["head_dim"] == 128:
        s[[5, 38, 77, 120]] = 10.0
    return s


def _prompt(c, seed, layer, b0, nb):
    """Prompt tensors of sequences b0 .. b0 + nb - 1: Q [nb][H*G][P][d], K and V [nb][H][P][d]."""
    H, G, d, P, dt = c["kv_heads"], c["q_per_kv"], c["head_dim"], c["hi"], _dtype(c)
    out = []
    for which, heads in ((0, H * G), (1, H), (2, H)):
        t = torch.empty((nb, heads, P, d), dtype=dt, device="cuda")
        for i in range(nb):
            x = _randn((heads, P, d), seed, ((layer * 512 + b0 + i) * 4 + which) * 8)
            t[i] = x * _key_scale(c) if which == 1 else x
        out.append(t)
    return out


def _tokens(c, seed, n=RING):
    """Decode inputs: q [n][b][H*G][d], k and v [n][b][H][d]."""
    b, H, G, d, dt = c["batch"], c["kv_heads"], c["q_per_kv"], c["head_dim"], _dtype(c)
    q = _randn((n, b, H * G, d), seed, 1, dt)
    k = (_randn((n, b, H, d), seed, 2) * _key_scale(c)).to(dt)
    return q, k, _randn((n, b, H, d), seed, 3, dt)


def _mlp(c, seed, layer):
    H, F, n_in = c["kv_heads"], c["scorer_hidden"], 3 * c["head_dim"]
    t = 10000 + layer * 16
    return {"W1": _randn((H, n_in, F), seed, t, scale=math.sqrt(2.0 / (n_in + F))),
            "b1": _randn((H, F), seed, t + 1, scale=0.1),
            "w2": _randn((H, F), seed, t + 2, scale=math.sqrt(2.0 / (F + 1))),
            "b2": _randn((H,), seed, t + 3, scale=0.1)}


def _mlstm(c, seed):
    H, n2, hh = c["kv_heads"], 2 * c["head_dim"], c["head_dim"] // 2
    std = {"Wq": math.sqrt(2.0 / (n2 + hh)), "wi": 1 / math.sqrt(n2), "a": math.sqrt(2.0 / (hh + 1))}
    w = {n: _randn((H, n2, hh), seed, 20000 + i, scale=std["Wq"]) for i, n in enumerate(("Wq", "Wk", "Wv"))}
    w.update({n: _randn((H, n2), seed, 20010 + i, scale=std["wi"]) for i, n in enumerate(("wi", "wf"))})
    w["a"] = _randn((H, hh), seed, 20020, scale=std["a"])
    w["bi"], w["b"] = torch.zeros(H, device="cuda"), torch.zeros(H, device="cuda")
    w["bf"] = torch.full((H,), 3.0, device="cuda")
    return w


def _projections(c, seed, layer):
    hid, d, Hq, H = c["hidden"], c["head_dim"], c["kv_heads"] * c["q_per_kv"], c["kv_heads"]
    shapes = {"Wq": (hid, Hq * d), "Wk": (hid, H * d), "Wv": (hid, H * d), "Wo": (Hq * d, hid)}
    out = {}
    for i, (n, s) in enumerate(shapes.items()):
        w = _randn(s, seed, 30000 + layer * 16 + i, scale=1 / math.sqrt(s[0]))
        out[n] = (w * _key_scale(c).repeat(H) if n == "Wk" else w).to(torch.bfloat16)
    return out


def _log_gamma(c):
    return torch.full((c["kv_heads"],), c["log_gamma"]) if c["log_gamma"] else None


def _cache(c, seed):
    kw = {"mlstm": _mlstm(c, seed)} if c["scorer"] == "mlstm" else dict(
        _mlp(c, seed, 0), log_gamma=_log_gamma(c), activation=c["scorer"])
    return kvpop.KVpopCache(c["batch"], c["kv_heads"], c["q_per_kv"], c["head_dim"], c["budget"],
                            c["window"], c["scorer_hidden"], _dtype(c), n_sink=c["sinks"], **kw)


def _prefill(c, seed, layer, cache, L):
    for b0 in range(0, c["batch"], GROUP):
        nb = min(GROUP, c["batch"] - b0)
        Q, K, V = _prompt(c, seed, layer, b0, nb)
        cache.prefill(Q, K, V, L[b0:b0 + nb], first_seq=b0)


# ---------------------------------------------------------------------- the passes
def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c, "i": 0, "L": _lengths(c, seed)}
    b, H, G, d, P = c["batch"], c["kv_heads"], c["q_per_kv"], c["head_dim"], c["hi"]
    dev = "cuda"
    if kind == "stack":
        layers = [dict(_projections(c, seed, l), **_mlp(c, seed, l)) for l in range(c["layers"])]
        stack = DecodeStack(layers, b, c["hidden"], H, G, d, c["budget"], c["window"],
                            c["scorer_hidden"], n_sink=c["sinks"])
        for l in range(c["layers"]):
            _prefill(c, seed, l, stack.caches[l], st["L"])
        st["xs"] = _randn((RING, b, c["hidden"]), seed, 4, torch.bfloat16)
        st["x"], st["y"] = torch.empty_like(st["xs"][0]), torch.empty_like(st["xs"][0])
        torch.matmul(st["xs"][0], layers[0]["Wq"])     # cuBLAS is set up before the capture
        stack.capture(st["x"], st["y"])
        st["stack"] = stack
        return st
    if kind in ("step", "prompt"):
        st["cache"] = _cache(c, seed)
    if kind == "step" or c["scorer"] == "mlstm":
        st["tok"] = _tokens(c, seed)
        st["out"] = torch.empty((b, H * G, d), device=dev)
        st["evict"] = torch.empty((b, H, 2), dtype=torch.int32, device=dev)
        st["score"] = torch.empty((b, H), device=dev)
    if kind == "step":
        _prefill(c, seed, 0, st["cache"], st["L"])
        return st
    st["Q"], st["K"], st["V"] = _prompt(c, seed, 0, 0, b)
    if kind == "prompt" and c["scorer"] != "mlstm":
        # rows past a sequence's length are left as they are
        st["Y"] = torch.zeros((b, H * G, P, d), device=dev)
        st["lse"] = torch.zeros((b, H * G, P), device=dev)
        st["rank"] = torch.empty((b, H, P), dtype=torch.int32, device=dev)
        st["tau"] = torch.empty_like(st["rank"])
    if kind == "train":
        st["prio"] = _randn((b * H, P), seed, 5)
    return st


def run(st):
    c, kind = st["case"], st["case"]["kind"]
    if kind == "stack":
        st["x"].copy_(st["xs"][st["i"] % RING])
        st["i"] += 1
        st["stack"].graph.replay()
        return {"hidden": st["y"]}
    if kind == "prompt" and c["scorer"] != "mlstm":
        st["cache"].prefill_attend(st["Q"], st["K"], st["V"], st["L"], st["Y"], lse=st["lse"],
                                   rank=st["rank"], tau=st["tau"])
        return {n: st[n] for n in ("Y", "lse", "rank", "tau")}
    if kind in ("step", "prompt"):
        if kind == "prompt":
            st["cache"].prefill(st["Q"], st["K"], st["V"], st["L"])
        j = st["i"] % RING
        st["i"] += 1
        q, k, v = st["tok"]
        st["cache"].step(q[j], k[j], v[j], st["out"], evict_info=st["evict"], score_out=st["score"])
        return {n: st[n] for n in ("out", "evict", "score")}
    Q, K, V = st["Q"], st["K"], st["V"]
    if kind == "target":
        lse = kvpop.causal_lse(Q, K)
        logm, target = kvpop.future_target(Q, K, lse, c["window"], lookahead=c["lookahead"],
                                           agg=c["agg"])
        return {"lse": lse, "logm": logm, "target": target}
    b, H, P = K.shape[:3]
    k = c["budget"] - c["sinks"]
    order = torch.empty((b * H, P), dtype=torch.int32, device=K.device)
    rank, tau = kvpop.topk_cutoff(st["prio"], c["sinks"], c["window"], k, order=order)
    Y, lse = kvpop.prompt_attention(Q, K, V, rank.view(b, H, P), tau.view(b, H, P), c["sinks"],
                                    c["window"], k, order=order)
    logm, target = kvpop.future_target(Q, K, lse, c["window"], lookahead=c["lookahead"],
                                       agg=c["agg"])
    return {"rank": rank, "tau": tau, "Y": Y, "lse": lse, "logm": logm, "target": target}


# ---------------------------------------------------------------------- what a pass cannot do without
def _masked_keys(P, c):
    """Retained keys summed over the queries of a prompt of P tokens."""
    most = c["budget"] + c["window"]
    n = min(P, most)
    return n * (n + 1) // 2 + max(0, P - most) * most


def work(case):
    c, kind = case, case["kind"]
    b, H, G, d = c["batch"], c["kv_heads"], c["q_per_kv"], c["head_dim"]
    esz = 4 if c["dtype"] == "f32" else 2
    mean = c["hi"] if c["lo"] == c["hi"] else (c["lo"] + c["hi"]) / 2
    pairs = b * H
    if c["scorer"] == "mlstm":
        weights = H * 2 * d * (3 * (d // 2) + 2)
    else:
        weights = H * c["scorer_hidden"] * (3 * d + 2)
    if kind in ("step", "stack"):
        keys = min(mean, c["budget"]) + c["window"]
        step_bytes = pairs * (keys * 2 * d * esz + (2 * G + 2) * d * esz) + weights * 4
        step_flops = pairs * (4 * G * d * keys) + 2 * weights * b
        if c["scorer"] == "mlstm":
            step_bytes += pairs * 2 * 4 * d * (d // 2 + 1)      # state read and written
            step_flops += pairs * 4 * d * (d // 2)
        if kind == "step":
            return {"bytes": step_bytes, "flops": step_flops}
        proj = c["hidden"] * (2 * H * G + 2 * H) * d
        return {"bytes": c["layers"] * (step_bytes + 2 * proj) + 4 * b * c["hidden"],
                "flops": c["layers"] * (step_flops + 2 * proj * b)}
    tokens = b * mean
    qkv = tokens * H * (G + 2) * d * esz
    if kind == "prompt":
        kept = b * min(mean, c["budget"])
        cache = kept * H * 2 * d * esz
        if c["scorer"] == "mlstm":
            hh = d // 2
            flops = tokens * H * (2 * 2 * d * (3 * hh + 2) + 4 * d * hh + 4 * d)
            return {"bytes": tokens * H * 2 * d * esz + 2 * cache + weights * 4, "flops": flops}
        flops = b * H * G * 4 * d * _masked_keys(int(mean), c) + 2 * tokens * weights
        return {"bytes": qkv + tokens * H * (G * (d + 1) * 4 + 8) + cache + weights * 4, "flops": flops}
    S = c["hi"]
    if kind == "target":
        reach = S if not c["lookahead"] else min(S, c["lookahead"])
        future = sum(min(max(0, S - t - c["window"]), reach) for t in range(S))
        return {"bytes": tokens * H * ((G + 1) * d * esz + (2 * G + 1) * 4),
                "flops": b * H * G * 2 * d * (S * (S + 1) // 2 + future)}
    future = sum(max(0, S - t - c["window"]) for t in range(S))
    return {"bytes": qkv + tokens * H * (4 * (G * d + 2 * G + 4)),
            "flops": b * H * G * (4 * d * _masked_keys(S, c) + 2 * d * future)}


# ---------------------------------------------------------------------- the same in 64 bits
def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))


def _score_mlp(w, h, x):
    return _gelu(x @ w["W1"][h].double() + w["b1"][h].double()) @ w["w2"][h].double() + w["b2"][h].double()


def _qbar(qm, D):
    """Mean over positions u+1 .. u+D of qm [T][d], for u = 0 .. T-D-1."""
    s = torch.cumsum(qm, 0)
    return (s[D:] - s[:-D]) / D


def _prompt_scores(c, w, h, Q, K, V):
    """fp64 scores of tokens 0 .. P-D-1 of one (sequence, head): Q [G][P][d], K, V [P][d]."""
    n = max(0, K.shape[0] - c["window"])
    if n == 0:
        return torch.empty(0, dtype=torch.float64, device=K.device)
    x = torch.cat([K[:n], V[:n], _qbar(Q.mean(0), c["window"])], 1)
    return torch.cat([_score_mlp(w, h, x[i:i + 65536]) for i in range(0, n, 65536)])


def _priority(c, score):
    u = torch.arange(score.numel(), dtype=torch.float32, device=score.device)
    return score.float() - u * c["log_gamma"]


def _kept(c, prio):
    """Positions in slot order (ascending) and their priorities."""
    s, B, n = c["sinks"], c["budget"], prio.numel()
    if n <= B:
        pos = torch.arange(n, device=prio.device)
    else:
        order = torch.argsort(prio[s:], descending=True, stable=True)[:B - s] + s
        pos = torch.cat([torch.arange(s, device=prio.device), order]).sort().values
    return pos, prio[pos]


def _step64(c, q, k, v, K, V, pos, prio, u, score):
    """Output [G][d] of the step that brings (k, v) to a sequence whose earlier keys and values
    are K and V, its slots holding `pos`; u leaves the window with `score`."""
    P, s, B = K.shape[0], c["sinks"], c["budget"]
    if u >= 0:
        r = score.float() - torch.tensor(float(u), device=K.device) * c["log_gamma"]
        if pos.numel() < B:
            pos = torch.cat([pos, torch.tensor([u], device=K.device)])
        else:
            at = int(torch.argmin(prio[s:])) + s
            if bool(r > prio[at]):
                pos = pos.clone()
                pos[at] = u
    keys = torch.cat([pos, torch.arange(max(0, P + 1 - c["window"]), P, device=K.device)])
    KK, VV = torch.cat([K[keys], k[None]]), torch.cat([V[keys], v[None]])
    return torch.softmax(q @ KK.T / math.sqrt(c["head_dim"]), -1) @ VV


def _layer64(c, seed, layer, w, L, q, k, v):
    """One decode step of a layer after its prompt: outputs [b][H*G][d] and scores [b][H]."""
    H, G, D = c["kv_heads"], c["q_per_kv"], c["window"]
    out = torch.empty_like(q)
    score = torch.full((c["batch"], H), math.nan, dtype=torch.float64, device="cuda")
    for b in range(c["batch"]):
        Qb, Kb, Vb = (t[0, :, :L[b]].double() for t in _prompt(c, seed, layer, b, 1))
        for h in range(H):
            Q, K, V = Qb[h * G:(h + 1) * G], Kb[h], Vb[h]
            qh, u = q[b, h * G:(h + 1) * G], L[b] - D
            if c["scorer"] == "mlstm":
                r = _mlstm64(w, h, D, torch.cat([K, k[b, h][None]]), torch.cat([V, v[b, h][None]]))
                prio = _priority(c, r[:max(0, u)])
                if u >= 0:
                    score[b, h] = r[u]
            else:
                prio = _priority(c, _prompt_scores(c, w, h, Q, K, V))
                if u >= 0:
                    qm = torch.cat([Q.mean(0)[u + 1:], qh.mean(0)[None]]).mean(0)
                    score[b, h] = _score_mlp(w, h, torch.cat([K[u], V[u], qm]))
            pos, kept = _kept(c, prio)
            out[b, h * G:(h + 1) * G] = _step64(c, qh, k[b, h], v[b, h], K, V, pos, kept, u, score[b, h])
    return out, score


def _hedgehog(y):
    return torch.cat([torch.softmax(y, -1), torch.softmax(-y, -1)], -1)


def _mlstm64(w, h, D, K, V):
    """fp64 scores of tokens 0 .. T-D-1 of one (sequence, head) with T tokens: the state that has
    absorbed tokens 0 .. u+D, read out with u's query.  Token t weighs its input gate times the
    forget gates after it."""
    g = lambda n: w[n][h].double()  # noqa: E731
    x = torch.cat([K, V], 1)
    T = x.shape[0]
    qt, kt, vt = _hedgehog(x @ g("Wq")), _hedgehog(x @ g("Wk")), x @ g("Wv")
    lf = torch.cumsum(torch.nn.functional.logsigmoid(x @ g("wf") + g("bf")), 0)
    gi = x @ g("wi") + g("bi")
    out = []
    for u0 in range(0, T - D, 1024):
        u = torch.arange(u0, min(T - D, u0 + 1024), device=x.device)
        n = int(u[-1]) + D + 1
        late = torch.arange(n, device=x.device)[None] > u[:, None] + D
        a = torch.exp((lf[u + D][:, None] - lf[None, :n] + gi[None, :n]).masked_fill_(late, -math.inf))
        a *= qt[u] @ kt[:n].T
        hh = (a @ vt[:n]) / a.sum(1, keepdim=True)
        out.append((hh * torch.sigmoid(hh)) @ g("a") + g("b"))
    return torch.cat(out) if out else torch.empty(0, dtype=torch.float64, device=x.device)


def _topk64(prio, n, P, s, D, k):
    """Ranks [P] and cutoffs [P] of one row whose tokens from n on have no priority."""
    p = torch.full((P,), -math.inf, device=prio.device)
    p[:n] = prio[:n]
    order = torch.argsort(p, descending=True, stable=True)
    rank = torch.empty(P, dtype=torch.int64, device=prio.device)
    rank[order] = torch.arange(P, device=prio.device)
    # the cutoff of q: the min(k, n_q)-th smallest rank of the tokens s .. q - D
    tau = torch.full((P,), -1, dtype=torch.int64, device=prio.device)
    for q0 in range(0, P, 512):
        q = torch.arange(q0, min(P, q0 + 512), device=prio.device)
        hi = int(q[-1]) - D + 1
        if hi <= s:
            continue
        t = torch.arange(s, hi, device=prio.device)
        r = torch.where(t[None] <= q[:, None] - D, rank[s:hi][None], P)
        many = (t[None] <= q[:, None] - D).sum(1)
        best = torch.sort(r, 1).values[:, :k]
        at = torch.clamp(many, max=k) - 1
        tau[q] = torch.where(many > 0, best.gather(1, at.clamp(min=0)[:, None])[:, 0], -1)
    return rank, tau


def _masked64(c, Q, K, V, rank, tau, k):
    """Outputs [G][P][d] and normalisers [G][P] under the running top-k mask."""
    G, P, d = Q.shape
    s, D = c["sinks"], c["window"]
    Y, lse = torch.empty_like(Q), torch.empty((G, P), dtype=torch.float64, device=Q.device)
    for q0 in range(0, P, 512):
        q = torch.arange(q0, min(P, q0 + 512), device=Q.device)
        n = int(q[-1]) + 1
        t = torch.arange(n, device=Q.device)
        gap = q[:, None] - t[None]
        ok = (gap >= 0) & ((t < s)[None] | (gap < D) | (rank[:n][None] <= tau[q][:, None]))
        x = (Q[:, q] @ K[:n].T / math.sqrt(d)).masked_fill_(~ok, -math.inf)
        lse[:, q] = torch.logsumexp(x, -1)
        Y[:, q] = torch.exp(x - lse[:, q, None]) @ V[:n]
    return Y, lse


def _future64(c, Q, K, lse):
    """Future log masses [G][S] and the target [S] of one (sequence, head)."""
    G, S, d = Q.shape
    w, la = c["window"], c["lookahead"]
    logm = torch.full((G, S), -math.inf, dtype=torch.float64, device=Q.device)
    for t0 in range(0, max(0, S - w), 512):
        t = torch.arange(t0, min(S - w, t0 + 512), device=Q.device)
        hi = S if not la else min(S, int(t[-1]) + w + la + 1)
        q = torch.arange(t0 + w, hi, device=Q.device)
        far = q[None] - t[:, None] - w
        ok = (far >= 0) & ((far <= la) if la else True)
        x = K[t] @ Q[:, q].transpose(1, 2) / math.sqrt(d) - lse[:, None, q]
        logm[:, t] = torch.logsumexp(x.masked_fill_(~ok, -math.inf), -1)
    n = torch.clamp(S - w - torch.arange(S, device=Q.device), min=1)
    n = torch.clamp(n, max=la + 1) if la else n
    mass = torch.exp(logm)
    mass = mass.max(0).values if c["agg"] == "max" else mass.mean(0)
    return logm, torch.log(1e-6 + mass / n)


def exact(case, seed):
    c, kind = case, case["kind"]
    H, G, d, P, D = c["kv_heads"], c["q_per_kv"], c["head_dim"], c["hi"], c["window"]
    L = _lengths(c, seed)
    with torch.no_grad():
        if kind == "stack":
            # fp64 products, rounded to bf16 where the stack stores them
            bf = lambda t: t.to(torch.bfloat16).double()  # noqa: E731
            x = _randn((RING, c["batch"], c["hidden"]), seed, 4, torch.bfloat16)[0].double()
            for l in range(c["layers"]):
                p, w = _projections(c, seed, l), _mlp(c, seed, l)
                q, k, v = (bf(x @ p[n].double()).view(c["batch"], -1, d) for n in ("Wq", "Wk", "Wv"))
                o, _ = _layer64(c, seed, l, w, L, q, k, v)
                x = bf(x + bf(bf(o).view(c["batch"], -1) @ p["Wo"].double()))
            return {"hidden": x}
        if kind in ("step", "prompt") and (kind == "step" or c["scorer"] == "mlstm"):
            q, k, v = (t[0].double() for t in _tokens(c, seed))
            w = _mlstm(c, seed) if c["scorer"] == "mlstm" else _mlp(c, seed, 0)
            out, score = _layer64(c, seed, 0, w, L, q, k, v)
            return {"out": out, "evict": None, "score": score}
        Q, K, V = _prompt(c, seed, 0, 0, c["batch"])
        if work(c)["flops"] > 8e12:
            return None
        if kind == "prompt":
            w, k = _mlp(c, seed, 0), c["budget"] - c["sinks"]
            Y = torch.zeros((c["batch"], H * G, P, d), dtype=torch.float64, device="cuda")
            lse = torch.zeros((c["batch"], H * G, P), dtype=torch.float64, device="cuda")
            for b in range(c["batch"]):
                n = L[b]
                for h in range(H):
                    g = slice(h * G, (h + 1) * G)
                    q64, k64, v64 = Q[b, g, :n].double(), K[b, h, :n].double(), V[b, h, :n].double()
                    prio = _priority(c, _prompt_scores(c, w, h, q64, k64, v64))
                    rank, tau = _topk64(prio, prio.numel(), n, c["sinks"], D, k)
                    Y[b, g, :n], lse[b, g, :n] = _masked64(c, q64, k64, v64, rank, tau, k)
            return {"Y": Y, "lse": lse, "rank": None, "tau": None}
        shape = (c["batch"], H * G, P)
        new = lambda *s: torch.empty(s, dtype=torch.float64, device="cuda")  # noqa: E731
        lse, logm, target = new(*shape), new(*shape), new(c["batch"], H, P)
        Y = new(*shape, d) if kind == "train" else None
        prio = _randn((c["batch"] * H, P), seed, 5) if kind == "train" else None
        for b in range(c["batch"]):
            for h in range(H):
                g = slice(h * G, (h + 1) * G)
                q64, k64, v64 = Q[b, g].double(), K[b, h].double(), V[b, h].double()
                if kind == "train":
                    k = c["budget"] - c["sinks"]
                    rank, tau = _topk64(prio[b * H + h], P, P, c["sinks"], D, k)
                    Y[b, g], lse[b, g] = _masked64(c, q64, k64, v64, rank, tau, k)
                else:
                    for q0 in range(0, P, 512):
                        n = min(P, q0 + 512)
                        x = q64[:, q0:n] @ k64[:n].T / math.sqrt(d)
                        later = torch.arange(n, device="cuda")[None] > torch.arange(q0, n, device="cuda")[:, None]
                        lse[b, g, q0:n] = torch.logsumexp(x.masked_fill_(later, -math.inf), -1)
                logm[b, g], target[b, h] = _future64(c, q64, k64, lse[b, g])
        if kind == "train":
            return {"rank": None, "tau": None, "Y": Y, "lse": lse, "logm": logm, "target": target}
        return {"lse": lse, "logm": logm, "target": target}
