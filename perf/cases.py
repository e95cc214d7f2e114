"""The calls that users of this library make, as timed cases.

A case is one pass through the public Python entry points on tensors that are already on the GPU:

* ``layer``    one attention layer: estimate -> select -> attention (``prefill_layer``), optionally fused with the
               previous layer's score, as in every layer of a stack but the first;
* ``project``  the same layer from its hidden states: Q / K / V projection with rotary embedding, whose epilogue already
               leaves the representatives, then the layer on them;
* ``varlen``   a packed batch of sequences of different lengths (``prefill_varlen``), in [tokens, heads, head_dim] storage;
* ``dense``    dense causal attention, the baseline of the method and what a stack runs in the layers it does not prune;
* ``decode``   block criticality and block list of the newest token against a key cache.

Q, K and V follow the recipe of ``paper_2409_12490_b200/inputs.py`` (clustered keys in runs, AR(1) queries that dwell on a
cluster), drawn on the device.
"""
from __future__ import annotations

import dataclasses
import math

import torch

from paper_2409_12490_b200 import CONFIGS
from paper_2409_12490_b200 import binding as cp

DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}
D_MODEL = 4096          # hidden size of the 32-head shapes (32 x 128)


# ---------------------------------------------------------------- the cases
def _case(path, tokens, dtype="bf16", batch=1, heads_q=32, heads_kv=8, head_dim=128, segment=512, block=32, budget=1024,
          fused=False, **more):
    return {"path": path, "tokens": tokens, "dtype": dtype, "batch": batch, "heads_q": heads_q, "heads_kv": heads_kv,
            "head_dim": head_dim, "segment": segment, "block": block, "budget": budget, "fused": fused, **more}


def _named(name, path="layer", **kw):
    """The shape of one of the repository's configurations."""
    c = CONFIGS[name]
    args = dict(tokens=c.seq_len, dtype=c.dtype, batch=c.batch, heads_q=c.n_q_heads, heads_kv=c.n_kv_heads,
                head_dim=c.head_dim, segment=c.segment_size, block=c.block_size, budget=c.budget_tokens)
    args.update(kw)
    return _case(path, **args)


def listed():
    return [
        # a small fp32 layer (configuration C1): checks, small models, anything that wants fp32
        {"name": "layer_1k_fp32", **_named("C1")},
        # a short prompt of odd length at the paper's segment / block / budget: launches and latency
        {"name": "layer_1300_ragged", **_case("layer", 1300)},
        # ordinary prompts: C2, and C3 as a layer inside a stack (fused with the previous layer's score)
        {"name": "layer_8k", **_named("C2")},
        {"name": "layer_32k_fused", **_named("C3", fused=True)},
        # the longest prompts: the headline layer C4, and the paper's own operating point in its own precision
        {"name": "layer_128k", **_named("C4")},
        {"name": "layer_128k_paper_fp16", **_named("paper_128k", dtype="f16", fused=True)},
        # 16-bit heads of 64 channels, two prompts of odd length at a time
        {"name": "layer_6k_hd64_fp16", **_case("layer", 6001, dtype="f16", batch=2, heads_q=16, heads_kv=4, head_dim=64, block=64)},
        # a serving batch of unequal prompts
        {"name": "varlen_8_prompts", **_case("varlen", 25739, lengths="731,4096,1502,9217,388,2750,6031,1024")},
        # a layer from its hidden states
        {"name": "project_layer_16k", **_case("project", 16384, block=64, budget=2048)},
        # an unpruned layer, length not a multiple of any tile
        {"name": "dense_20k", **_case("dense", 20001)},
        # the next token of a short and of a long conversation
        {"name": "decode_8k", **_case("decode", 8191)},
        {"name": "decode_128k", **_case("decode", 130001, block=128, budget=4096)},
    ]


def draw(rng):
    path = rng.choice(["layer"] * 9 + ["varlen"] * 3 + ["project"] * 2 + ["dense"] * 3 + ["decode"] * 3)
    dtype = rng.choice(["bf16", "bf16", "f16"])
    heads_q, heads_kv = rng.choice([(32, 8), (32, 8), (32, 4), (16, 4), (8, 2), (8, 8)])
    head_dim, batch, more = 128, 1, {}
    segment = rng.choice([128, 256, 512, 512, 1024])
    block = rng.choice([b for b in (32, 64, 128) if b <= segment])
    budget = rng.choice([b for b in (1024, 2048, 4096, 8192) if b >= segment]) if rng.random() < 0.8 else block * rng.randint(segment // block, 64)
    low, high = 300, 131072
    if path == "layer" and rng.random() < 0.35:                  # fp32, or heads of 64 channels
        dtype = rng.choice(["f32", "f32", "bf16", "f16"])
        head_dim = 64 if dtype != "f32" else rng.choice([64, 128])
        high = 4096 if dtype == "f32" else 16384
        heads_q, heads_kv = rng.choice([(4, 2), (8, 2)]) if dtype == "f32" else rng.choice([(16, 4), (32, 8)])
    elif path == "dense":
        high = 24576
    elif path == "project":
        high, heads_q, heads_kv = 32768, 32, rng.choice([8, 4])
    tokens = int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))
    if rng.random() < 0.25:
        tokens = max(256, tokens // 256 * 256)
    if path in ("layer", "decode") and tokens <= 16384:
        batch = rng.choice([1, 1, 2, 3])
    if path == "varlen":
        lens = [int(round(math.exp(rng.uniform(math.log(100), math.log(12000))))) for _ in range(rng.randint(2, 16))]
        more["lengths"] = ",".join(map(str, lens))
        tokens = sum(lens)
    c = _case(path, tokens, dtype, batch, heads_q, heads_kv, head_dim, segment, block, budget,
              fused=path == "layer" and rng.random() < 0.5, **more)
    while _too_large(c):
        c["tokens"] = c["tokens"] * 3 // 5
    return c


def _too_large(c):
    """More work than the largest listed case of its kind."""
    if c["path"] == "varlen" or c["path"] == "decode":
        return False
    rows = c["tokens"] * c["batch"] * c["heads_q"]
    scores = c["batch"] * c["heads_q"] * (c["tokens"] / c["segment"]) * (c["tokens"] / c["block"])
    keys = c["tokens"] / 2 if c["path"] == "dense" else min(c["budget"], c["tokens"] / 2)
    if c["dtype"] == "f32" or c["head_dim"] == 64:
        return rows * keys * c["head_dim"] > 2 * 6001 * 16 * 1024 * 64
    return rows * keys > 131072 * 32 * 4096 or scores > 32 * 256 * 4096


# ---------------------------------------------------------------- inputs
def _runs(gen, heads, n, lo, hi, n_ids):
    """ids[head, t], constant over runs whose lengths are uniform in [lo, hi]."""
    m = n // lo + 2
    ends = torch.randint(lo, hi + 1, (heads, m), generator=gen, device="cuda").cumsum(1)
    ids = torch.randint(0, n_ids, (heads, m), generator=gen, device="cuda")
    at = torch.arange(n, device="cuda").expand(heads, n).contiguous()
    return ids.gather(1, torch.searchsorted(ends, at, right=True))


def _ar1(x, rho):
    """y[t] = rho * y[t-1] + x[t] along dim 0, by doubling (terms below 1e-6 left out)."""
    step = 1
    while rho ** step > 1e-6 and step < x.shape[0]:
        y = x.clone()
        y[step:] += rho ** step * x[:-step]
        x, step = y, 2 * step
    return x


def _qkv(c, seed, tokens, batch, layer=0):
    """Q [B,Hq,n,d], K and V [B,Hkv,n,d]: keys in runs of one cluster, queries walking towards a cluster they dwell on."""
    n, d, hq, hkv, dt = tokens, c["head_dim"], c["heads_q"], c["heads_kv"], DTYPES[c["dtype"]]
    rho = 0.98 if n > 65536 else 0.95
    clusters = 256 if n > 65536 else (64 if n > 4096 else 8)
    struct = torch.Generator(device="cuda").manual_seed(seed)             # the layers of a stack share runs and dwells
    value = torch.Generator(device="cuda").manual_seed(seed * 64 + 17 + layer)
    normal = lambda *s: torch.randn(*s, generator=value, device="cuda")
    Q = torch.empty((batch, hq, n, d), dtype=dt, device="cuda")
    K = torch.empty((batch, hkv, n, d), dtype=dt, device="cuda")
    V = torch.empty_like(K)
    for b in range(batch):
        z = _runs(struct, hkv, n, c["block"], 4 * c["block"], clusters)
        w = _runs(struct, hq, n, 2 * c["segment"], 6 * c["segment"], clusters)
        for h in range(hkv):
            centres = normal(clusters, d)
            K[b, h] = centres[z[h]] + 0.3 * normal(n, d)
            V[b, h] = normal(n, d)
            for q in range(h * (hq // hkv), (h + 1) * (hq // hkv)):
                x = (1 - rho) * centres[w[q]] + 0.5 * math.sqrt(1 - rho * rho) * normal(n, d)
                x[0] = centres[w[q, 0]]
                Q[b, q] = _ar1(x, rho)
    return Q, K, V


def _problem(c, tokens, **kw):
    return cp.Problem(c["batch"], c["heads_q"], c["heads_kv"], tokens, c["head_dim"], c["segment"], c["block"],
                      max(c["budget"], c["segment"]) // c["block"], DTYPES[c["dtype"]], **kw)


def prepare(case, seed):
    c, n = case, case["tokens"]
    if c["path"] == "varlen":
        lens = [int(x) for x in c["lengths"].split(",")]
        prob = _problem(c, max(lens))
        parts = [_qkv(c, seed * 32 + i, m, 1) for i, m in enumerate(lens)]
        pack = lambda k: torch.cat([p[k][0].transpose(0, 1) for p in parts]).transpose(0, 1)    # storage [tokens, heads, d]
        cu = [0]
        for m in lens:
            cu.append(cu[-1] + m)
        return {"path": c["path"], "prob": prob, "ws": cp.alloc_workspace(prob), "cu": cu, "Q": pack(0), "K": pack(1), "V": pack(2)}
    prob = _problem(c, n)
    state = {"path": c["path"], "prob": prob, "ws": cp.alloc_workspace(prob)}
    if c["path"] == "project":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        normal = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(prob.dtype)
        # hidden states of neighbouring tokens resemble each other; weights of scale 1 / sqrt(d_model) keep Q, K, V at unit scale
        walk = torch.randn((n, D_MODEL), generator=gen, device="cuda")
        state["X"] = (_ar1(walk, 0.9) * math.sqrt(1 - 0.81)).to(prob.dtype).view(c["batch"], n, D_MODEL)
        for name, heads in (("Wq", c["heads_q"]), ("Wk", c["heads_kv"]), ("Wv", c["heads_kv"])):
            state[name] = normal(heads * c["head_dim"], D_MODEL) / math.sqrt(D_MODEL)
        half = c["head_dim"] // 2
        angle = torch.outer(torch.arange(n, device="cuda").double(), 500000.0 ** (-torch.arange(half, device="cuda").double() / half))
        state["cos"], state["sin"] = angle.cos().float(), angle.sin().float()
        state["ready"] = dataclasses.replace(prob, flags=cp.FLAG_SUMMARIES_READY)
        return state
    Q, K, V = _qkv(c, seed, n, c["batch"])
    if c["path"] == "decode":
        state.update(q_last=Q[:, :, -1].contiguous(), K=K)
        return state
    state.update(Q=Q, K=K, V=V, S_prev=None)
    if c["fused"]:
        Q0, K0, _ = _qkv(c, seed, n, c["batch"], layer=1)
        state["S_prev"] = cp.estimate(prob, Q0, K0, state["ws"])
    return state


# ---------------------------------------------------------------- one pass
def run(state):
    path, prob, ws = state["path"], state["prob"], state["ws"]
    if path == "layer":
        return cp.prefill_layer(prob, state["Q"], state["K"], state["V"], ws, S_prev=state["S_prev"])
    if path == "project":
        Q, K, V = cp.project_qkv(prob, state["X"], state["Wq"], state["Wk"], state["Wv"], ws, rope_cos=state["cos"], rope_sin=state["sin"])
        return (Q, K, V) + cp.prefill_layer(state["ready"], Q, K, V, ws)
    if path == "varlen":
        O, _, idx, cnt, S_flat = cp.prefill_varlen(prob, state["cu"], state["Q"], state["K"], state["V"], ws)
        return O, idx, cnt, S_flat
    if path == "dense":
        return cp.dense_attention(prob, state["Q"], state["K"], state["V"], ws)
    S = cp.decode_estimate(prob, state["q_last"], state["K"], ws)
    return (S,) + cp.decode_select(prob, S, ws)


# ---------------------------------------------------------------- what a pass cannot do without
def _layer_work(c, n):
    """(bytes, flops) of estimate + select + attention for one sequence: each tensor once; the score products of the
    blocks a segment can see and the attention products of the keys a row attends to."""
    es = 4 if c["dtype"] == "f32" else 2
    B, hq, hkv, d, seg, blk = c["batch"], c["heads_q"], c["heads_kv"], c["head_dim"], c["segment"], c["block"]
    k = max(c["budget"], seg) // blk
    r, n1, n2 = seg // blk, -(-n // seg), -(-n // blk)
    scores = pairs = 0
    for j in range(n1):
        rows = min(seg, n - j * seg)
        vis = min(n2, (j + 1) * r)
        past = max(0, min(k, vis) - (vis - j * r)) * blk
        scores += vis
        pairs += rows * past + rows * (rows + 1) // 2
    nbytes = es * B * n * d * (2 * hq + 2 * hkv) + B * hq * (8 * n1 * n2 * (2 if c["fused"] else 1) + 4 * n1 * (k + 1))
    return nbytes, B * hq * d * (8 * scores + 4 * pairs)


def work(case):
    c, n = case, case["tokens"]
    es = 4 if c["dtype"] == "f32" else 2
    B, hq, hkv, d = c["batch"], c["heads_q"], c["heads_kv"], c["head_dim"]
    if c["path"] == "varlen":
        parts = [_layer_work(c, int(x)) for x in c["lengths"].split(",")]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if c["path"] == "dense":
        return {"bytes": es * B * n * d * (2 * hq + 2 * hkv), "flops": 4 * B * hq * d * n * (n + 1) // 2}
    if c["path"] == "decode":
        n2 = -(-n // c["block"])
        k = max(c["budget"], c["segment"]) // c["block"]
        return {"bytes": es * B * d * (n * hkv + hq) + B * hq * (8 * n2 + 4 * (k + 1)), "flops": 4 * B * hq * d * n2}
    nbytes, flops = _layer_work(c, n)
    if c["path"] == "project":
        out = (hq + 2 * hkv) * d
        nbytes += es * (B * n * D_MODEL + out * D_MODEL + B * n * out) + 4 * n * d - es * B * n * d * (hq + 2 * hkv)   # Q, K, V are counted once
        flops += 2 * B * n * D_MODEL * out
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times what two correct evaluations were seen to differ by: the tensor-core kernels against the SIMT kernel
    with unrounded probabilities for 16-bit types (bf16: rel 2.5e-3, max 0.041; fp16: rel 3.2e-4, max 5.5e-3), the SIMT
    kernel against fp64 for fp32 (rel 1.8e-6, max 4.1e-5).  Scores are fp64 on exact inputs; decode returns nothing else.
    Q, K and V of ``project`` round differently for another order of the same sums (rel 1.5e-4); their scores then differ in
    the fourth digit, 0.1 % of the lists' entries change, and a row whose list changed may attend to other keys altogether
    (O: rel 0.015, max 2.3), so there the bounds are as wide as can be stated."""
    if case["path"] == "decode":
        return {"rel": 1e-11, "max": 1e-9, "differ": 1e-3}
    if case["path"] == "project":
        return {"rel": 0.03, "max": 0.99, "differ": 5e-3}
    if case["dtype"] == "f32":
        return {"rel": 7e-6, "max": 1.6e-4, "differ": 1e-3}
    return {"rel": 1.3e-3, "max": 0.022, "differ": 1e-3} if case["dtype"] == "f16" else {"rel": 1e-2, "max": 0.16, "differ": 1e-3}
