"""Performance cases of the DAS-Wave hot path: what a decoding engine calls, per
step, through the package's public entry points.

A case is a dict of plain values.  `op` names the path:
  attend   the attention calls of one draft or verify pass over `layers` core
           layers (das_mature_v_attention, AttentionCall, das_verify_attention
           or das_mature_v_attention_f8),
  accept   das_greedy_accept of `groups` micro-batches,
  readout  das_wave_readout of one refinement round of `groups` micro-batches,
  commit   das_kv_append / das_kv_append_f8,
  cycle    one whole speculative step: draft, verify, accept and commit.

`how` says how a program issues the calls: "call" (the plain function, its
outputs allocated), "object" (arguments checked once, outputs kept; the
function with its outputs given where there is no such object) or "graph"
(the step captured once in a CUDA graph, as latency-bound loops do, and
replayed).

Sizes are those of the workloads in synth/workloads.py, of the tests, or
generic.  An attention case's cache holds the depths that its calls read
(two, instead of all R) in the layout of the full one, so that several states
fit the device.  Lengths come from the case alone (`lens`), values from the
seed.
"""
import math
import random

import numpy as np
import torch

import paper_2609_34538_gb300 as das

BF16 = torch.bfloat16


# ---- cases ---------------------------------------------------------------------
def _attend(name, **kw):
    c = dict(name=name, op="attend", kind="draft", store="bf16", how="object", batch=1, layers=2,
             q_heads=32, kv_heads=8, head_dim=128, prefix_lo=4096, prefix_hi=4096, block_lo=16,
             block_hi=16, lens=1)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call: one draft layer of a small looped model, issued
        # directly.  What it costs is latency and launches.
        _attend("tiny_call", how="call", layers=1, q_heads=4, kv_heads=4, head_dim=64,
                prefix_lo=256, prefix_hi=256, block_lo=4, block_hi=4),
        # Interactive single-sequence decoding (a 3.5B-class looped model): a
        # draft step's four core layers in a graph.
        _attend("decode_step", how="graph", layers=4, kv_heads=32, block_lo=8, block_hi=8),
        # Batched serving of math / code prompts: ragged prefixes and blocks.
        _attend("batched_step", batch=16, layers=4, prefix_lo=1024, prefix_hi=8192, block_lo=4),
        # Long-context drafting, the largest step.
        _attend("long_step", batch=4, prefix_lo=32768, prefix_hi=32768),
        # The verifier's pass over 16 candidates of 8 sequences.
        _attend("verify_step", kind="verify", batch=8, prefix_lo=16384, prefix_hi=16384),
        # A model with 64-wide heads, ragged prefixes of odd lengths.
        _attend("ragged_d64", batch=8, head_dim=64, prefix_lo=501, prefix_hi=12001, block_lo=7),
        # Mature-V over a cache that keeps its shallow depths as e4m3: e4m3
        # keys, bf16 values.
        _attend("e4m3_draft", store="e4m3", batch=4, prefix_lo=16384, prefix_hi=16384),
        # A verify pass at a depth below R of that cache: keys and values
        # e4m3 (31 of the 32 depths of every verify pass).
        _attend("e4m3_verify", store="e4m3", kind="verify", batch=8, prefix_lo=2003,
                prefix_hi=12001, block_lo=13, block_hi=13),
        # Greedy acceptance after a verify pass of 8 sequences.
        dict(name="accept_b8", op="accept", how="graph", batch=8, width=16, vocab=32000, groups=4,
             lens=1),
        # A late, wide round of a refinement over an odd vocabulary.
        dict(name="readout_odd", op="readout", how="graph", batch=4, width=25, vocab=50257,
             groups=4, lens=1),
        # Commit of a verify pass at all 32 depths into an e4m3 cache.
        dict(name="commit_e4m3", op="commit", store="e4m3", how="graph", batch=8, layers=4,
             kv_heads=8, head_dim=128, depths=32, capacity=256, width=16, lens=1),
        # One whole speculative step of two sequences: draft and verify over
        # four layers, acceptance, commit at every depth.
        dict(name="cycle", op="cycle", how="graph", batch=2, layers=4, q_heads=32, kv_heads=8,
             head_dim=128, depths=8, capacity=2100, prefix_lo=1024, prefix_hi=2048, width=8,
             vocab=32000, lens=1),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.random()
    lens = rng.randrange(1 << 20)
    if kind < 0.7:
        store = "e4m3" if rng.random() < 0.35 else "bf16"
        D = 64 if rng.random() < 0.3 else 128
        G = rng.choice([1, 1, 2, 4, 4, 8])
        T = _log_int(rng, 1, min(32, 64 // G))
        H = rng.choice([2, 4, 8, 8, 16, 32])
        B = _log_int(rng, 1, 48)
        hi = _log_int(rng, 32, 32768)
        layers = rng.choice([1, 2, 4])
        # no larger than the largest listed case
        while B * hi * layers * H * D > 4 * 32768 * 2 * 8 * 128:
            hi = max(32, hi // 2)
            B = max(1, B * 2 // 3)
        ragged = rng.random() < 0.6
        c = dict(op="attend", kind="verify" if rng.random() < 0.35 else "draft", store=store,
                 how=rng.choice(["graph", "object", "object"]), batch=B, layers=layers,
                 q_heads=H * G, kv_heads=H, head_dim=D, prefix_lo=max(1, hi // 8) if ragged else hi,
                 prefix_hi=hi, block_lo=max(1, T // 2) if ragged else T, block_hi=T, lens=lens)
        return c
    if kind < 0.8:
        return dict(op="accept", how=rng.choice(["graph", "call"]), batch=_log_int(rng, 1, 24),
                    width=rng.choice([1, 3, 4, 8, 15, 16]),
                    vocab=rng.choice([32000, 32003, 50257, _log_int(rng, 1000, 131072)]),
                    groups=rng.choice([1, 2, 4]), lens=lens)
    if kind < 0.9:
        return dict(op="readout", how=rng.choice(["graph", "call"]), batch=_log_int(rng, 1, 16),
                    width=rng.randrange(2, 33),
                    vocab=rng.choice([32000, 50257, _log_int(rng, 1000, 131072)]), groups=2,
                    lens=lens)
    return dict(op="commit", store=rng.choice(["bf16", "e4m3"]),
                how=rng.choice(["graph", "call"]), batch=_log_int(rng, 1, 16),
                layers=rng.choice([1, 2, 4]), kv_heads=rng.choice([4, 8]),
                head_dim=rng.choice([64, 128]), depths=rng.choice([4, 8, 32]), capacity=256,
                width=rng.randrange(2, 33), lens=lens)


# ---- lengths (from the case alone) ---------------------------------------------
def _lengths(case):
    r = random.Random(case["lens"])
    n = case["batch"]
    P = [r.randint(case["prefix_lo"], case["prefix_hi"]) for _ in range(n)]
    lo = case.get("block_lo", case.get("width"))
    hi = case.get("block_hi", case.get("width"))
    T = [r.randint(lo, hi) for _ in range(n)]
    T[r.randrange(n)] = hi  # the buffers' rows are the longest block's
    return P, T


def _accepted(case):
    """Planted acceptance lengths, 0 .. width."""
    r = random.Random(case["lens"] + 7)
    return [r.randint(0, case["width"]) for _ in range(case["batch"])]


def _commit_prefix(case):
    r = random.Random(case["lens"] + 9)
    return [r.randint(1, case["capacity"] - case["width"]) for _ in range(case["batch"])]


# ---- inputs --------------------------------------------------------------------
def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 64 + what)
    return g


def _i32(v):
    return torch.tensor(v, dtype=torch.int32, device="cuda")


def _normal(shape, g):
    return torch.randn(shape, generator=g, device="cuda", dtype=BF16)


def _depths_of(case):
    """(key slot, value slot) of the two-depth cache: slot 1 is a shallow
    depth, slot 2 full depth R.  Drafts read keys at the shallow depth and
    values at R (Mature-V); the verifier reads one depth for both: R, or on an
    e4m3 cache a depth below R."""
    if case["kind"] == "draft":
        return 1, 2
    return (1, 1) if case["store"] == "e4m3" else (2, 2)


def _matured(top, noise, g):
    """A shallow depth of `top`: the mature value plus what is still missing."""
    x = torch.randn(top.shape, generator=g, device="cuda", dtype=BF16)
    return x.mul_(noise).add_(top)


def _to_e4m3(x):
    return x.clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)


def _queries(shape, g):
    """Query rows of differing sharpness (score deviations of about 0.5 to 3)."""
    q = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    s = torch.rand(shape[:-1] + (1,), generator=g, device="cuda")
    return (q * torch.exp(1.8 * s - 0.7)).to(BF16)


def _blocks(case, T, seed, what):
    """q, k_blk, v_blk of one layer call."""
    B, D = case["batch"], case["head_dim"]
    g = _gen(seed, what)
    return (_queries((B, T, case["q_heads"], D), g), _normal((B, T, case["kv_heads"], D), g),
            _normal((B, T, case["kv_heads"], D), g))


def _outputs(q):
    B, T, H, _ = q.shape
    return torch.empty_like(q), torch.empty((B, H, T), dtype=torch.float32, device="cuda")


def _capture(step):
    """The step as a CUDA graph (one eager pass first: library set-up)."""
    step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    return graph


def _prepare_attend(case, seed):
    B, L, H, D = case["batch"], case["layers"], case["kv_heads"], case["head_dim"]
    P, T = _lengths(case)
    rows, cap = max(T), max(P) + max(T)
    kslot, vslot = _depths_of(case)
    top = (L, B, cap, H, D)
    s = {"case": case, "P": P, "T": T, "prefix_len": _i32(P), "block_len": _i32(T)}
    k_top, v_top = _normal(top, _gen(seed, 0)), _normal(top, _gen(seed, 1))
    if case["store"] == "bf16":
        low_k = _matured(k_top, 0.7, _gen(seed, 2)) if kslot == 1 else k_top
        low_v = _matured(v_top, 0.8, _gen(seed, 3)) if vslot == 1 else v_top
        s["cache"] = das.DepthKVCache(torch.stack([low_k, k_top]), torch.stack([low_v, v_top]))
        s["ws"] = das.new_workspace(s["cache"], case["q_heads"], rows)
    else:
        low_k = _to_e4m3(_matured(k_top, 0.7, _gen(seed, 2)))[None].contiguous()
        low_v = _to_e4m3(_matured(v_top, 0.8, _gen(seed, 3)))[None].contiguous()
        s["cache"] = das.DepthKVCacheF8(k_top, v_top, low_k, low_v)
        s["ws"] = das.new_workspace_f8(s["cache"], case["q_heads"], rows)
    s["in"] = [_blocks(case, rows, seed, 8 + l) for l in range(L)]
    if case["how"] != "call":
        s["out"] = [_outputs(x[0]) for x in s["in"]]
        if case["store"] == "bf16":
            s["calls"] = [das.AttentionCall(s["cache"], s["prefix_len"], s["block_len"], *x,
                                            s["ws"], out=o, lse=l)
                          for x, (o, l) in zip(s["in"], s["out"])]
    if case["how"] == "graph":
        s["graph"] = _capture(lambda: _step_attend(s))
    return s


def _step_attend(s):
    case = s["case"]
    kd, vd = _depths_of(case)
    got = []
    for l in range(case["layers"]):
        if case["how"] == "call":
            got.append(das.das_mature_v_attention(s["cache"], l, kd, vd, s["prefix_len"],
                                                  s["block_len"], *s["in"][l], s["ws"])
                       if case["store"] == "bf16" else
                       das.das_mature_v_attention_f8(s["cache"], l, kd, vd, s["prefix_len"],
                                                     s["block_len"], *s["in"][l], s["ws"]))
        elif case["store"] == "e4m3":
            o, lse = s["out"][l]
            got.append(das.das_mature_v_attention_f8(s["cache"], l, kd, vd, s["prefix_len"],
                                                     s["block_len"], *s["in"][l], s["ws"], out=o,
                                                     lse=lse))
        elif kd == vd:
            got.append(s["calls"][l].verify(l, kd))
        else:
            got.append(s["calls"][l].mature_v(l, kd, vd))
    return got


def _logits(case, seed, what):
    """fp32 logits and draft ids whose first `accepted` proposals agree."""
    B, W, V = case["batch"], case["width"], case["vocab"]
    x = torch.randn((B, W, V), generator=_gen(seed, what), device="cuda").mul_(2.0)
    draft = x.argmax(-1).to(torch.int32)
    for b, a in enumerate(_accepted(case)):
        if a < W:
            draft[b, a] = (draft[b, a] + 1) % V
    return x, draft


def _prepare_accept(case, seed):
    s = {"case": case, "in": [_logits(case, seed, 8 + i) for i in range(case["groups"])]}
    if case["how"] == "graph":
        B, W = case["batch"], case["width"]
        s["out"] = [tuple(torch.zeros(n, dtype=torch.int32, device="cuda") for n in (B, (B, W), B))
                    for _ in range(case["groups"])]
        s["graph"] = _capture(lambda: _step_accept(s))
    return s


def _step_accept(s):
    if "out" not in s:
        return [das.das_greedy_accept(x, d) for x, d in s["in"]]
    return [das.das_greedy_accept(x, d, *o) for (x, d), o in zip(s["in"], s["out"])]


def _prepare_readout(case, seed):
    B, W = case["batch"], case["width"]
    s = {"case": case, "in": [_logits(case, seed, 8 + i)[0] for i in range(case["groups"])]}
    # the anchors, then the window's guesses, which the readout revises in place
    s["out"] = [torch.zeros((B, W + 1), dtype=torch.int32, device="cuda") for _ in s["in"]]
    for i, t in enumerate(s["out"]):
        t[:, 0] = torch.arange(B, device="cuda", dtype=torch.int32) + 100 * i
    if case["how"] == "graph":
        s["graph"] = _capture(lambda: _step_readout(s))
    return s


def _step_readout(s):
    return [das.das_wave_readout(x, t) for x, t in zip(s["in"], s["out"])]


def _staged(case, seed):
    shape = (case["depths"], case["layers"], case["batch"], case["width"], case["kv_heads"],
             case["head_dim"])
    return _normal(shape, _gen(seed, 4)), _normal(shape, _gen(seed, 5))


def _prepare_commit(case, seed):
    R, top = case["depths"], (case["layers"], case["batch"], case["capacity"], case["kv_heads"],
                              case["head_dim"])
    if case["store"] == "bf16":
        cache = das.DepthKVCache(_normal((R,) + top, _gen(seed, 0)), _normal((R,) + top, _gen(seed, 1)))
    else:
        code = lambda what: torch.randint(0, 120, (R - 1,) + top, generator=_gen(seed, what),
                                          dtype=torch.uint8, device="cuda")
        cache = das.DepthKVCacheF8(_normal(top, _gen(seed, 0)), _normal(top, _gen(seed, 1)),
                                   code(2), code(3))
    base = _i32(_commit_prefix(case))
    s = {"case": case, "cache": cache, "new": _staged(case, seed), "base": base,
         "accepted": _i32(_accepted(case)), "prefix_len": base.clone(),
         "flag": torch.zeros(1, dtype=torch.int32, device="cuda")}
    if case["how"] == "graph":
        s["out"] = _step_commit(s)
        s["graph"] = _capture(lambda: _step_commit(s))
    return s


def _step_commit(s):
    s["prefix_len"].copy_(s["base"])  # the sequences stand where they stood before the step
    if s["case"]["store"] == "bf16":
        das.das_kv_append(s["cache"], *s["new"], s["accepted"], s["prefix_len"], s["flag"])
        parts = (s["cache"].k, s["cache"].v)
    else:
        das.das_kv_append_f8(s["cache"], *s["new"], s["accepted"], s["prefix_len"], s["flag"])
        parts = (s["cache"].k_top, s["cache"].v_top, s["cache"].k_low, s["cache"].v_low)
    return {"cache": parts, "prefix_len": s["prefix_len"], "flag": s["flag"]}


def _prepare_cycle(case, seed):
    P, T = _lengths(case)
    shape = (case["depths"], case["layers"], case["batch"], case["capacity"], case["kv_heads"],
             case["head_dim"])
    cache = das.DepthKVCache(_normal(shape, _gen(seed, 0)), _normal(shape, _gen(seed, 1)))
    base = _i32(P)
    s = {"case": case, "cache": cache, "base": base, "prefix_len": base.clone(),
         "block_len": _i32(T), "new": _staged(case, seed),
         "flag": torch.zeros(1, dtype=torch.int32, device="cuda"),
         "ws": das.new_workspace(cache, case["q_heads"], case["width"]),
         "logits": _logits(case, seed, 7)}
    s["in"] = {k: [_blocks(case, case["width"], seed, 8 + 16 * i + l) for l in range(case["layers"])]
               for i, k in enumerate(("draft", "verify"))}
    s["out"] = {k: [_outputs(x[0]) for x in s["in"][k]] for k in s["in"]}
    s["calls"] = {k: [das.AttentionCall(cache, s["prefix_len"], s["block_len"], *x, s["ws"], out=o,
                                        lse=l) for x, (o, l) in zip(s["in"][k], s["out"][k])]
                  for k in s["in"]}
    B, W = case["batch"], case["width"]
    s["accept"] = tuple(torch.zeros(n, dtype=torch.int32, device="cuda") for n in (B, (B, W), B))
    s["graph"] = _capture(lambda: _step_cycle(s))
    return s


def _step_cycle(s):
    R = s["case"]["depths"]
    s["prefix_len"].copy_(s["base"])  # the sequences stand where they stood before the step
    for l, call in enumerate(s["calls"]["draft"]):
        call.mature_v(l, 2, R)
    for l, call in enumerate(s["calls"]["verify"]):
        call.verify(l, R)
    das.das_greedy_accept(*s["logits"], *s["accept"])
    das.das_kv_append(s["cache"], *s["new"], s["accept"][0], s["prefix_len"], s["flag"])
    return {"draft": s["out"]["draft"], "verify": s["out"]["verify"], "accept": s["accept"],
            "cache": (s["cache"].k, s["cache"].v), "prefix_len": s["prefix_len"], "flag": s["flag"]}


_PREPARE = {"attend": _prepare_attend, "accept": _prepare_accept, "readout": _prepare_readout,
            "commit": _prepare_commit, "cycle": _prepare_cycle}
_STEP = {"attend": _step_attend, "accept": _step_accept, "readout": _step_readout,
         "commit": _step_commit, "cycle": _step_cycle}


def prepare(case, seed):
    return _PREPARE[case["op"]](case, seed)


def run(state):
    if "graph" not in state:
        return _STEP[state["case"]["op"]](state)
    state["graph"].replay()
    if state["case"]["op"] != "cycle":
        return state["out"]
    return {"draft": state["out"]["draft"], "verify": state["out"]["verify"],
            "accept": state["accept"], "cache": (state["cache"].k, state["cache"].v),
            "prefix_len": state["prefix_len"], "flag": state["flag"]}


# ---- work ----------------------------------------------------------------------
def _attend_work(case, P, T, rows, key_bytes, value_bytes):
    """One layer call."""
    B, Hq, H, D = case["batch"], case["q_heads"], case["kv_heads"], case["head_dim"]
    nbytes = sum(P) * H * D * (key_bytes + value_bytes)
    nbytes += B * rows * D * 2 * (2 * Hq + 2 * H) + B * Hq * rows * 4
    flops = sum(4.0 * t * (p + (t + 1) / 2) * Hq * D for p, t in zip(P, T))
    return nbytes, flops


def _commit_bytes(case, accepted, low_bytes):
    rows = sum(min(a + 1, case["width"]) for a in accepted)
    per_depth = 2 * rows * case["layers"] * case["kv_heads"] * case["head_dim"]
    return per_depth * (2 * case["depths"] + low_bytes * (case["depths"] - 1) + 2)


def work(case):
    op = case["op"]
    if op == "attend":
        P, T = _lengths(case)
        kd, vd = _depths_of(case)
        size = lambda d: 1 if case["store"] == "e4m3" and d == 1 else 2
        b, f = _attend_work(case, P, T, max(T), size(kd), size(vd))
        return {"bytes": b * case["layers"], "flops": f * case["layers"]}
    if op == "commit":
        low = 1 if case["store"] == "e4m3" else 2
        return {"bytes": _commit_bytes(case, _accepted(case), low), "flops": 0}
    row = case["vocab"] * 4 * case["batch"]
    if op == "accept":
        return {"bytes": case["groups"] * case["width"] * (row + 8 * case["batch"]), "flops": 0}
    if op == "readout":
        return {"bytes": case["groups"] * case["width"] * (row + 4 * case["batch"]), "flops": 0}
    P, T = _lengths(case)
    b, f = _attend_work(case, P, T, case["width"], 2, 2)
    return {"bytes": 2 * case["layers"] * b + case["width"] * row +
            _commit_bytes(case, _accepted(case), 2), "flops": 2 * case["layers"] * f}


# ---- exact values --------------------------------------------------------------
def _exact_call(case, k, v, P, T, q, kb, vb):
    """(out, lse) in float64; k, v [B][cap][H][D] of the depths that are read."""
    B, rows, Hq, D = q.shape
    H = kb.shape[2]
    G = Hq // H
    out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    lse = torch.full((B, Hq, rows), -math.inf, dtype=torch.float64, device="cuda")
    for b in range(B):
        p, t = P[b], T[b]
        if t == 0:
            continue
        K = torch.cat([k[b, :p].double(), kb[b, :t].double()]).permute(1, 0, 2)
        V = torch.cat([v[b, :p].double(), vb[b, :t].double()]).permute(1, 0, 2)
        Q = q[b, :t].double().reshape(t, H, G, D).permute(1, 2, 0, 3).reshape(H, G * t, D)
        s = torch.matmul(Q, K.transpose(1, 2)) / math.sqrt(D)
        i = torch.arange(t, device="cuda").repeat(G)
        s[:, :, p:].masked_fill_(torch.arange(t, device="cuda")[None, :] > i[:, None], -math.inf)
        l = torch.logsumexp(s, -1)
        o = torch.matmul(torch.exp(s - l[..., None]), V)
        out[b, :t] = o.reshape(H, G, t, D).permute(2, 0, 1, 3).reshape(t, Hq, D)
        lse[b, :, :t] = l.reshape(Hq, t)
    return out, lse


def _first_argmax(x):
    m = x.double().max(-1, keepdim=True).values
    pos = torch.arange(x.shape[-1], device="cuda", dtype=torch.float64)
    return torch.where(x.double() == m, pos, math.inf).min(-1).values.to(torch.int32)


def _exact_accept(x, draft):
    t = _first_argmax(x)
    B, W = t.shape
    acc = (draft == t).int().cumprod(1).sum(1).to(torch.int32)
    at = acc.long().clamp(max=W - 1)[:, None]
    nxt = torch.where(acc < W, t.gather(1, at)[:, 0], draft[:, -1])
    return acc, t, nxt


def _exact_commit(parts, new, accepted, base, width, low):
    """The cache tensors (copies) after the commit; `low`: codes of the depths
    below R follow the two bf16 tensors of depth R."""
    parts = [x.clone() for x in parts]
    for b, (a, p) in enumerate(zip(accepted, base)):
        n = min(a + 1, width)
        for i, x in enumerate(new):
            rows = x[:, :, b, :n]
            if low:
                parts[i][:, b, p:p + n] = rows[-1]
                parts[2 + i][:, :, b, p:p + n] = _to_e4m3(rows[:-1])
            else:
                parts[i][:, :, b, p:p + n] = rows
    return tuple(parts)


def exact(case, seed):
    s = _PREPARE[case["op"]](dict(case, how="call"), seed) if case["op"] != "cycle" else \
        _PREPARE["cycle"](case, seed)
    op = case["op"]
    if op == "attend":
        kd, vd = _depths_of(case)
        got = []
        for l in range(case["layers"]):
            if case["store"] == "bf16":
                k, v = s["cache"].k[kd - 1, l], s["cache"].v[vd - 1, l]
            else:
                c, f8 = s["cache"], torch.float8_e4m3fn
                k = c.k_low[0, l].view(f8).to(BF16) if kd == 1 else c.k_top[l]
                v = c.v_low[0, l].view(f8).to(BF16) if vd == 1 else c.v_top[l]
            got.append(_exact_call(case, k, v, s["P"], s["T"], *s["in"][l]))
        return got
    if op == "accept":
        return [_exact_accept(x, d) for x, d in s["in"]]
    if op == "readout":
        return [torch.cat([t[:, :1], _first_argmax(x)], 1) for x, t in zip(s["in"], s["out"])]
    if op == "commit":
        low, c = case["store"] == "e4m3", s["cache"]
        base, accepted = _commit_prefix(case), _accepted(case)
        parts = (c.k_top, c.v_top, c.k_low, c.v_low) if low else (c.k, c.v)
        n = np.minimum(np.array(accepted) + 1, case["width"])
        return {"cache": _exact_commit(parts, s["new"], accepted, base, case["width"], low),
                "prefix_len": _i32((np.array(base) + n).tolist()), "flag": s["flag"]}
    # the cycle: the seed's cache anew (preparing the step has run it once)
    P, T = _lengths(case)
    R, W = case["depths"], case["width"]
    shape = s["cache"].shape
    k, v = _normal(shape, _gen(seed, 0)), _normal(shape, _gen(seed, 1))
    got = {name: [_exact_call(case, k[kd - 1, l], v[R - 1, l], P, T, *s["in"][name][l])
                  for l in range(case["layers"])] for name, kd in (("draft", 2), ("verify", R))}
    acc = _exact_accept(*s["logits"])
    accepted = acc[0].tolist()
    n = np.minimum(np.array(accepted) + 1, W)
    got.update(accept=acc, cache=_exact_commit((k, v), s["new"], accepted, P, W, False),
               prefix_len=_i32((np.array(P) + n).tolist()), flag=torch.zeros_like(s["flag"]))
    return got
