"""The work that a program using this library has it do, as measurable cases.

Every case goes through the library's public entry points
(``paper_2509_01190_gb300.zsaa``).  Shapes are those of the repository's own
configurations (``inputs.py``: the 1B and 8B decoder shapes, the classifier, the
float32 configuration) or generic ones.  Whole models run a stack of 6 or 8 of
their layers: bf16 storage noise grows with depth, and at full depth it is as
large as what a comparison of logits could allow; every layer's width, head
count, vocabulary, batch and length are the real ones.

Kinds of case:

* ``generate``    pruned prefill into a KV cache, then decode steps on given
                  tokens; returns every step's logits (steps = 0: prefill alone).
* ``classify``    pruned prefill with the classifier head; ``ragged`` batches run
                  as one packed variable-length call.
* ``float32``     the float32 path: the whole pruned forward with the LM head.
* ``attention``   one pruning layer's attention and its soft-score column mass.
* ``projections`` the four projections of one layer at a given number of rows.
* ``select``      isolated score + top-k + compaction.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2509_01190_gb300 import zsaa as z

SHAPE_1B = dict(d=2048, heads=32, kv_heads=8, hd=64, ffn=8192, vocab=128256)
SHAPE_8B = dict(d=4096, heads=32, kv_heads=8, hd=128, ffn=14336, vocab=128256)
RMS_EPS = 1e-5
CLASSES = 4


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # Serving: a batch of prompts, pruned 4x, then tokens generated on the
        # pruned cache (the repository's own decode benchmark, half the layers).
        dict(name="generate_1b_b8", kind="generate", layers=8, B=8, L=512, accel=4.0, steps=16, **SHAPE_1B),
        # One interactive request: latency of a short prompt and its first tokens.
        dict(name="generate_1b_b1", kind="generate", layers=8, B=1, L=99, accel=2.0, steps=12, **SHAPE_1B),
        # Long-prompt prefill of the largest configuration (time to first token).
        dict(name="prefill_8b_b4", kind="generate", layers=6, B=4, L=2048, accel=3.0, steps=0, **SHAPE_8B),
        # Throughput classification of many short texts, pruned 3x.
        dict(name="classify_1b_b64", kind="classify", layers=8, B=64, L=256, accel=3.0, ragged=False, **SHAPE_1B),
        # The same of texts of different lengths in one packed call.
        dict(name="classify_ragged_1b", kind="classify", layers=8, B=16, L=700, accel=3.0, ragged=True, **SHAPE_1B),
        # The float32 configuration: the smallest call, launch latency counts.
        dict(name="float32_tiny", kind="float32", layers=2, B=2, L=64, accel=2.0, rate=True,
             d=128, heads=4, kv_heads=4, hd=32, ffn=512, vocab=1000),
        # A float32 model of ordinary size (checking a bf16 deployment against 32 bits).
        dict(name="float32_d1024", kind="float32", layers=4, B=4, L=384, accel=2.0, rate=False,
             d=1024, heads=16, kv_heads=4, hd=64, ffn=4096, vocab=8000),
        # A pruning layer's attention and column mass at the largest configuration.
        dict(name="attention_8b_n2048", kind="attention", B=4, N=2048, heads=32, kv_heads=8, hd=128, causal=True),
        # An encoder without grouped heads (every query head has its own keys),
        # a length that no tile divides.
        dict(name="attention_encoder_mha", kind="attention", B=16, N=501, heads=16, kv_heads=16, hd=64, causal=False),
        # A deep layer's projections, on the few hundred rows that pruning leaves.
        dict(name="projections_8b_m360", kind="projections", M=360, **SHAPE_8B),
        # Isolated selection over a large hidden state (the repository's microbenchmark).
        dict(name="select_b32_l4096", kind="select", B=32, L=4096, d=4096, k=1024, f32=False),
        # The same on one small float32 batch of odd length, scores returned.
        dict(name="select_f32_small", kind="select", B=3, L=1537, d=1152, k=385, f32=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["generate", "classify", "float32", "attention", "projections", "select"])
    if kind == "generate":
        if rng.random() < 0.3:
            shape, layers, B, L, least = SHAPE_8B, rng.randint(2, 6), _log_int(rng, 1, 4), _log_int(rng, 64, 2048), 3.0
        else:
            shape, layers, B, L, least = SHAPE_1B, rng.randint(2, 8), _log_int(rng, 1, 16), _log_int(rng, 16, 512), 1.3
        return dict(kind=kind, layers=layers, B=B, L=L, accel=round(rng.uniform(least, 6.0), 2),
                    steps=rng.randint(0, 16), **shape)
    if kind == "classify":
        B = _log_int(rng, 1, 64)
        return dict(kind=kind, layers=rng.randint(2, 8), B=B, L=_log_int(rng, 16, min(900, 16384 // B)),
                    accel=round(rng.uniform(2.5, 11.0), 2), ragged=rng.random() < 0.5, **SHAPE_1B)
    if kind == "float32":
        heads = rng.choice([4, 8, 16])
        kv = heads // rng.choice([1, 2, 4])
        hd = rng.choice([32, 64])
        return dict(kind=kind, layers=rng.randint(1, 4), B=_log_int(rng, 1, 4), L=_log_int(rng, 16, 384),
                    accel=round(rng.uniform(1.0, 4.0), 2), rate=rng.random() < 0.5, d=64 * rng.randint(2, 16),
                    heads=heads, kv_heads=kv, hd=hd, ffn=64 * rng.randint(4, 64), vocab=rng.randint(500, 8000))
    if kind == "attention":
        hd, kv, per = rng.choice([64, 128]), rng.choice([1, 2, 4, 8]), rng.choice([1, 2, 3, 4, 8])
        N = _log_int(rng, 1, 2048)
        most = 4 * 2048 * 2048 * 32 // (N * N * kv * per)
        return dict(kind=kind, B=_log_int(rng, 1, max(1, min(32, most))), N=N, heads=kv * per, kv_heads=kv, hd=hd,
                    causal=rng.random() < 0.6)
    if kind == "projections":
        return dict(kind=kind, M=_log_int(rng, 1, 4096), **rng.choice([SHAPE_1B, SHAPE_8B]))
    L, d = _log_int(rng, 16, 4096), 8 * _log_int(rng, 16, 512)
    return dict(kind="select", B=_log_int(rng, 1, 32), L=L, d=d, k=max(1, int(L / rng.uniform(1.0, 11.0))),
                f32=rng.random() < 0.4)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, *size, scale=0.02, dtype=torch.bfloat16):
    return (torch.randn(*size, generator=g, device="cuda") * scale).to(dtype)


def _weights(c, g):
    """Random-init weights as the repository draws them: N(0, 0.02), norm weights 1."""
    dt = torch.float32 if c["kind"] == "float32" else torch.bfloat16
    d, dq, dkv = c["d"], c["heads"] * c["hd"], c["kv_heads"] * c["hd"]
    one = torch.ones(d, device="cuda", dtype=dt)
    layers = [dict(attn_norm=one, wq=_normal(g, dq, d, dtype=dt), wk=_normal(g, dkv, d, dtype=dt),
                   wv=_normal(g, dkv, d, dtype=dt), wo=_normal(g, d, dq, dtype=dt), mlp_norm=one,
                   wg=_normal(g, c["ffn"], d, dtype=dt), wu=_normal(g, c["ffn"], d, dtype=dt),
                   wd=_normal(g, d, c["ffn"], dtype=dt)) for _ in range(c["layers"])]
    head = _normal(g, CLASSES if c["kind"] == "classify" else c["vocab"], d, dtype=dt)
    return dict(embed=_normal(g, c["vocab"], d, dtype=dt), layers=layers, final_norm=one, head=head)


def _theta(c):
    return 10000.0 if c["kind"] == "float32" else 500000.0


def _config(c):
    f32 = c["kind"] == "float32"
    prune = [1] if c.get("rate") else range(1, c["layers"])  # all layers but the last, or the first alone
    return z.make_config(c["layers"], c["d"], c["heads"], c["kv_heads"], c["hd"], c["ffn"], c["vocab"],
                         n_classes=CLASSES if c["kind"] == "classify" else 0, rope_theta=_theta(c), rms_eps=RMS_EPS,
                         dtype="f32" if f32 else "bf16", prune_layers=[p for p in prune if p <= c["layers"]],
                         plan_mode="rate" if c.get("rate") else "cost")


def _lengths(c, seed):
    """Lengths of a batch: all L, or for a ragged one spread from L/8 to L."""
    if not c.get("ragged"):
        return [c["L"]] * c["B"]
    r = np.random.default_rng(seed)
    return [int(n) for n in r.integers(max(1, c["L"] // 8), c["L"] + 1, size=c["B"])]


def _tokens(g, vocab, *size):
    return torch.randint(0, vocab, size, generator=g, device="cuda", dtype=torch.int32)


def _model_inputs(c, seed):
    g = _gen(seed)
    w = _weights(c, g)
    lengths = _lengths(c, seed)
    prompt = _tokens(g, c["vocab"], sum(lengths))
    following = _tokens(g, c["vocab"], max(1, c.get("steps", 0)), c["B"])
    return w, lengths, prompt, following


def _qkv(c, seed):
    # queries and keys after RoPE: N(0, 1), so that the soft-scores have some spread
    return _normal(_gen(seed), c["B"] * c["N"], (c["heads"] + 2 * c["kv_heads"]) * c["hd"], scale=1.0)


def _projection_inputs(c, seed):
    g = _gen(seed)
    d, dq, dkv, F, M = c["d"], c["heads"] * c["hd"], c["kv_heads"] * c["hd"], c["ffn"], c["M"]
    return dict(x=_normal(g, M, d, scale=1.0), o=_normal(g, M, dq, scale=0.3), a=_normal(g, M, F, scale=0.5),
                h=_normal(g, M, d, scale=1.0), wqkv=_normal(g, dq + 2 * dkv, d), wo=_normal(g, d, dq),
                wg=_normal(g, F, d), wu=_normal(g, F, d), wd=_normal(g, d, F),
                pos=torch.arange(M, device="cuda", dtype=torch.int32) * 3 % 4096)


def _hidden(c, seed):
    g = _gen(seed)
    scale = torch.exp(torch.randn(c["B"], c["L"], 1, generator=g, device="cuda"))  # log-normal row scales
    x = torch.randn(c["B"], c["L"], c["d"], generator=g, device="cuda") * scale
    return x if c["f32"] else x.to(torch.bfloat16)


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(case=c)
    if kind in ("generate", "classify", "float32"):
        w, lengths, prompt, following = _model_inputs(c, seed)
        s["model"] = z.Model(_config(c), w, c["B"], max(lengths))
        s["prompt"], s["lengths"] = prompt, lengths
        if kind == "generate":
            s["cache"] = z.Cache(s["model"], c["B"], c["L"], c["accel"], max(1, c["steps"]))
            s["following"] = following
            s["token"] = torch.empty(c["B"], device="cuda", dtype=torch.int32)
            s["next"] = torch.empty(c["B"], c["vocab"], device="cuda")
            s["logits"] = torch.empty(1 + c["steps"], c["B"], c["vocab"], device="cuda")
        elif kind == "classify":
            s["logits"] = torch.empty(c["B"], CLASSES, device="cuda")
        else:
            n = z.zsaa_plan(s["model"], c["L"], c["accel"])[0][-1]
            s["logits"] = torch.empty(c["B"], n, c["vocab"], device="cuda")
            s["kept"] = torch.empty(c["B"], n, device="cuda", dtype=torch.int32)
    elif kind == "attention":
        rows, N = c["B"] * c["N"], c["N"]
        s["qkv"] = _qkv(c, seed)
        s["out"] = torch.empty(rows, c["heads"] * c["hd"], device="cuda", dtype=torch.bfloat16)
        s["lse"] = torch.empty(c["B"], c["heads"], N, device="cuda")
        s["mass"] = torch.empty(c["B"], c["kv_heads"], N, device="cuda")
    elif kind == "projections":
        s.update(_projection_inputs(c, seed))
        new = dict(device="cuda", dtype=torch.bfloat16)
        s["out"] = (torch.empty(c["M"], s["wqkv"].shape[0], **new), torch.empty(c["M"], c["d"], **new),
                    torch.empty(c["M"], c["ffn"], **new), torch.empty(c["M"], c["d"], **new))
    else:
        s["hidden"] = _hidden(c, seed)
        s["idx"] = torch.empty(c["B"], c["k"], device="cuda", dtype=torch.int32)
        s["rows"] = torch.empty(c["B"], c["k"], c["d"], device="cuda", dtype=s["hidden"].dtype)
        s["scores"] = torch.empty(c["B"], c["L"], device="cuda")
    return s


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "generate":
        z.zsaa_prefill(s["model"], s["cache"], s["prompt"], s["logits"][0])
        for t in range(c["steps"]):
            s["token"].copy_(s["following"][t])
            z.zsaa_decode_step(s["model"], s["cache"], s["token"], s["next"])
            s["logits"][t + 1].copy_(s["next"])
        return s["logits"]
    if kind == "classify":
        if c["ragged"]:
            z.zsaa_forward_varlen(s["model"], s["prompt"], s["lengths"], c["accel"], s["logits"])
        else:
            z.zsaa_forward(s["model"], s["prompt"], c["B"], c["L"], c["accel"], s["logits"])
        return s["logits"]
    if kind == "float32":
        z.zsaa_forward(s["model"], s["prompt"], c["B"], c["L"], c["accel"], s["logits"], s["kept"])
        return s["logits"], s["kept"]
    if kind == "attention":
        size = (c["B"], c["N"], c["heads"], c["kv_heads"], c["hd"], z.ZSAA_BF16, c["causal"])
        z.zsaa_op_attention_ex(s["qkv"], *size, s["out"], s["lse"])
        z.zsaa_op_colmass_ex(s["qkv"], s["lse"], *size, s["mass"])
        return s["out"], s["lse"], s["mass"]
    if kind == "projections":
        M, d, dq, F = c["M"], c["d"], c["heads"] * c["hd"], c["ffn"]
        qkv, ho, act, hd = s["out"]
        z.zsaa_op_linear(s["x"], s["wqkv"], None, None, qkv, M, qkv.shape[1], d, z.ZSAA_BF16, z.EPI_ROPE,
                         s["pos"], dq + c["kv_heads"] * c["hd"], c["hd"], 500000.0)
        z.zsaa_op_linear(s["o"], s["wo"], None, s["h"], ho, M, d, dq, z.ZSAA_BF16, z.EPI_RESID)
        z.zsaa_op_linear(s["x"], s["wg"], s["wu"], None, act, M, F, d, z.ZSAA_BF16, z.EPI_SWIGLU)
        z.zsaa_op_linear(s["a"], s["wd"], None, s["h"], hd, M, d, F, z.ZSAA_BF16, z.EPI_RESID)
        return qkv, ho, act, hd
    if c["f32"]:
        z.zsaa_score_select_ex(s["hidden"], c["B"], c["L"], c["d"], z.ZSAA_F32, c["k"], z.ZSAA_FLAG_FORCE_KEEP_LAST,
                               None, s["scores"], s["idx"], s["rows"])
        return s["idx"], s["rows"], s["scores"]
    z.zsaa_score_select(s["hidden"], c["B"], c["L"], c["d"], c["k"], s["idx"], s["rows"])
    return s["idx"], s["rows"]


# ------------------------------------------------------------------ what a pass cannot do without

def _schedules(c, lengths):
    """Kept rows N_0..N_n of every sequence (Eq. 2, floor of 5 rows): the rate is
    1/accel, or the largest one whose modelled work is at most 1/accel of the
    unpruned batch's (60 bisection steps)."""
    n, d, dq, dkv, F = c["layers"], c["d"], c["heads"] * c["hd"], c["kv_heads"] * c["hd"], c["ffn"]
    prune = {1} if c.get("rate") else set(range(1, n))
    per_row = 2 * d * (dq + 2 * dkv) + 2 * dq * d + 6 * d * F

    def sched(L, alpha):
        out = [L]
        for layer in range(1, n + 1):
            prev = out[-1]
            out.append(min(prev, max(math.floor(alpha * prev), min(5, prev))) if layer in prune else prev)
        return out

    def cost(alpha):
        total = 0
        for L in lengths:
            s = sched(L, alpha)
            total += sum(m * per_row + 2 * m * m * dq for m in s[:-1])
            total += 2 * d * CLASSES if c["kind"] == "classify" else s[-1] * 2 * d * c["vocab"]
        return total

    if c.get("rate"):
        alpha = 1.0 / c["accel"]
    elif c["accel"] == 1.0:
        alpha = 1.0
    else:
        target, lo, hi = cost(1.0) / c["accel"], 0.0, 1.0
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if cost(mid) <= target else (lo, mid)
        alpha = lo
    return [sched(L, alpha) for L in lengths]


def work(case):
    c, kind = case, case["kind"]
    if kind == "attention":
        pairs = c["B"] * c["heads"] * (c["N"] * (c["N"] + 1) // 2 if c["causal"] else c["N"] ** 2)
        rows = c["B"] * c["N"]
        # inputs and outputs once; Q K^T and P V of the attention, Q K^T again of the column mass
        return dict(bytes=rows * ((2 * c["heads"] + 2 * c["kv_heads"]) * c["hd"] * 2 + (c["heads"] + c["kv_heads"]) * 4),
                    flops=6 * pairs * c["hd"])
    if kind == "select":
        e = 4 if c["f32"] else 2
        return dict(bytes=c["B"] * (c["L"] * c["d"] * e + c["k"] * (c["d"] * e + 4) + (4 * c["L"] if c["f32"] else 0)),
                    flops=2 * c["B"] * c["L"] * c["d"])
    d, dq, dkv, F = c["d"], c["heads"] * c["hd"], c["kv_heads"] * c["hd"], c["ffn"]
    attn_w, mlp_w = d * (2 * dq + 2 * dkv), 3 * d * F
    if kind == "projections":
        M = c["M"]
        return dict(bytes=2 * (attn_w + mlp_w + M * (2 * d + dq + F) + M * (dq + 2 * dkv + 2 * d + F)),
                    flops=2 * M * (attn_w + mlp_w))
    e = 4 if kind == "float32" else 2
    scheds = _schedules(c, _lengths(c, 0))
    n, flops, nbytes = c["layers"], 0, 0
    for s in scheds:
        for layer in range(n):
            m, kept = s[layer], s[layer + 1]
            flops += 2 * m * attn_w + 2 * kept * mlp_w + 4 * dq * (m * (m + 1) // 2)
            if kept < m:
                flops += 2 * dq * (m * (m + 1) // 2)
    weights = n * (attn_w + mlp_w) * e
    rows = sum(s[0] for s in scheds)
    nbytes += weights + rows * d * e
    if kind == "generate":
        passes = 1 + c["steps"]
        flops += passes * c["B"] * 2 * d * c["vocab"] + c["steps"] * c["B"] * n * 2 * (attn_w + mlp_w)
        kv = sum(2 * dkv * e * sum(s[:-1]) for s in scheds)  # the cache a step reads
        nbytes += c["steps"] * (weights + kv) + passes * c["vocab"] * (d * e + c["B"] * 4)
    elif kind == "classify":
        nbytes += c["B"] * CLASSES * 4
    else:
        out = sum(s[-1] for s in scheds)
        flops += 2 * out * d * c["vocab"]
        nbytes += c["vocab"] * d * e + out * c["vocab"] * 4
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    kind = case["kind"]
    if kind in ("generate", "classify"):
        # bf16 storage points of up to 8 layers, and selections between rows
        # whose scores are closer than that
        return {"rel": 0.03}
    if kind == "float32":
        return {"rel": 1e-5, "differ": 0.0}
    if kind == "select":
        return {"rel": 1e-6, "differ": 0.0}  # copied rows; 32-bit sums of squares
    return {"rel": 8e-3}  # one rounding to bf16 of 32-bit sums


# ------------------------------------------------------------------ the same in 64 bits

def _rms(x, w):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + RMS_EPS) * w


def _rope(x, pos, theta):
    """x [rows, heads, hd] rotated at pos [rows]: dims c and c + hd/2 are a pair."""
    half = x.shape[-1] // 2
    inv = theta ** (-2.0 * torch.arange(half, device=x.device, dtype=torch.float64) / (2 * half))
    ang = pos.double()[:, None, None] * inv
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * ang.cos() - b * ang.sin(), b * ang.cos() + a * ang.sin()], -1)


def _attend(q, k, v, causal):
    """q [n, Hq, hd], k and v [m, Hkv, hd] -> out [n, Hq, hd], log2 normaliser
    [Hq, n] and column mass [Hkv, m]."""
    n, Hq, hd = q.shape
    m, G = k.shape[0], k.shape[1]
    out, lse, mass = torch.empty_like(q), q.new_empty(Hq, n), q.new_zeros(G, m)
    hidden = torch.ones(n, m, device=q.device, dtype=torch.bool).triu(1 + m - n) if causal else None
    for g in range(G):  # one group at a time bounds the memory
        hs = slice(g * (Hq // G), (g + 1) * (Hq // G))
        sc = torch.einsum("nhd,md->hnm", q[:, hs], k[:, g]) / math.sqrt(hd)
        if causal:
            sc.masked_fill_(hidden, -math.inf)
        l = torch.logsumexp(sc, -1)
        p = torch.exp(sc - l[..., None])
        out[:, hs] = torch.einsum("hnm,md->nhd", p, v[:, g])
        lse[hs] = l / math.log(2.0)
        mass[g] = p.sum((0, 1))
    return out, lse, mass


def _heads(c, x, w, pos):
    """Rotated queries and keys, and values, of rows x."""
    q = (x @ w["wq"].T).view(len(x), c["heads"], c["hd"])
    k = (x @ w["wk"].T).view(len(x), c["kv_heads"], c["hd"])
    v = (x @ w["wv"].T).view(len(x), c["kv_heads"], c["hd"])
    return _rope(q, pos, _theta(c)), _rope(k, pos, _theta(c)), v


def _mlp(h, w):
    x = _rms(h, w["mlp_norm"])
    return h + (torch.nn.functional.silu(x @ w["wg"].T) * (x @ w["wu"].T)) @ w["wd"].T


def _exact_model(c, seed):
    w, lengths, prompt, following = _model_inputs(c, seed)
    scheds = _schedules(c, lengths)
    tokens = prompt.split(lengths)
    h = [w["embed"][t.long()].double() for t in tokens]
    pos = [torch.arange(n, device="cuda") for n in lengths]
    new = [w["embed"][t.long()].double() for t in following]  # rows of each decode step
    steps = c.get("steps", 0)
    kv = [[None] * c["layers"] for _ in lengths]
    for li, lw in enumerate(w["layers"]):
        lw = {k: v.double() for k, v in lw.items()}
        for b, n in enumerate(lengths):
            q, k, v = _heads(c, _rms(h[b], lw["attn_norm"]), lw, pos[b])
            out, _, mass = _attend(q, k, v, True)
            h[b] = h[b] + out.flatten(1) @ lw["wo"].T
            kv[b][li] = (k, v)
            keep = scheds[b][li + 1]
            if keep < len(h[b]):  # rows of the largest contribution, the last one always among them
                score = (mass * v.norm(dim=-1).T).sum(0)
                score[-1] = math.inf
                idx = torch.sort(torch.argsort(score, descending=True, stable=True)[:keep]).values
                h[b], pos[b] = h[b][idx], pos[b][idx]
            h[b] = _mlp(h[b], lw)
        for t in range(steps):  # a step's rows see the kept rows and the steps before
            x = _rms(new[t], lw["attn_norm"])
            q, k, v = _heads(c, x, lw, torch.full((c["B"],), c["L"] + t, device="cuda"))
            o = []
            for b in range(c["B"]):
                kv[b][li] = (torch.cat([kv[b][li][0], k[b:b + 1]]), torch.cat([kv[b][li][1], v[b:b + 1]]))
                o.append(_attend(q[b:b + 1], *kv[b][li], False)[0].flatten(1))
            new[t] = _mlp(new[t] + torch.cat(o) @ lw["wo"].T, lw)
    norm, head = w["final_norm"].double(), w["head"].double()
    if c["kind"] == "float32":
        return torch.stack([_rms(x, norm) @ head.T for x in h]), torch.stack(pos).int()
    last = torch.stack([x[-1] for x in h])
    if c["kind"] == "classify":
        return _rms(last, norm) @ head.T
    return torch.stack([_rms(x, norm) @ head.T for x in [last] + new[:steps]])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("generate", "classify", "float32"):
        if work(c)["flops"] > 1.2e13:  # over 20 s in 64 bits
            return None
        return _exact_model(c, seed)
    if kind == "attention":
        qkv = _qkv(c, seed).double().view(c["B"], c["N"], -1, c["hd"])
        H, G = c["heads"], c["kv_heads"]
        got = [_attend(x[:, :H], x[:, H:H + G], x[:, H + G:], c["causal"]) for x in qkv]
        return (torch.cat([o.flatten(1) for o, _, _ in got]), torch.stack([l for _, l, _ in got]),
                torch.stack([m for _, _, m in got]))
    if kind == "projections":
        s = {k: v.double() for k, v in _projection_inputs(c, seed).items()}
        M, hd = c["M"], c["hd"]
        qkv = (s["x"] @ s["wqkv"].T).view(M, -1, hd)
        r = c["heads"] + c["kv_heads"]
        qkv[:, :r] = _rope(qkv[:, :r], s["pos"], 500000.0)
        act = torch.nn.functional.silu(s["x"] @ s["wg"].T) * (s["x"] @ s["wu"].T)
        return qkv.flatten(1), s["h"] + s["o"] @ s["wo"].T, act, s["h"] + s["a"] @ s["wd"].T
    x = _hidden(c, seed)
    scores = torch.stack([r.double().norm(dim=-1) for r in x])
    order = scores.clone()
    if c["f32"]:
        order[:, -1] = math.inf  # the last position is always kept
    idx = torch.sort(torch.argsort(order, dim=1, descending=True, stable=True)[:, :c["k"]], dim=1).values
    rows = torch.gather(x, 1, idx[..., None].expand(-1, -1, c["d"])).double()
    return (idx.int(), rows, scores) if c["f32"] else (idx.int(), rows)
