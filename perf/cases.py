"""Workloads of the library, from the smallest calls to the largest: prefill (span-search followed by
span-attention), chunks of a chunked prefill, the per-span mode with a local window, decode steps, and
prefill through host buffers.  Shapes are those of ``synth.CONFIGS`` and of the tests, or lie between
them.

Inputs are i.i.d. N(0,1) as in ``synth.py``, with planted key spans where a case says so.  Routing
queries and keys are rounded to multiples of 1/64: every product is then a multiple of 2^-12 and a score
stays below 2^9, so that fp32 sums of the products are exact in any order and the selection (and with it
everything downstream of a near-tie) does not depend on the order of summation.
"""
import math

import numpy as np
import torch

import paper_2601_18401_b200 as sla
from paper_2601_18401_b200 import synth

DEV = "cuda:0"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _prefill(name, rows, pos0=0, batch=1, q_heads=32, kv_heads=8, head_dim=128, dtype="bf16", top_k=8, span_len=0,
             planted=0):
    return {"name": name, "kind": "prefill", "batch": batch, "q_heads": q_heads, "kv_heads": kv_heads,
            "head_dim": head_dim, "dtype": dtype, "rows": rows, "pos0": pos0, "top_k": top_k, "span_len": span_len,
            "back": 2, "fwd": 0, "window": 0, "planted": planted}


def _decode(name, n_ctx, batch=1, q_heads=32, kv_heads=4, head_dim=128, dtype="bf16", top_k=16, span_len=0,
            gated=False):
    return {"name": name, "kind": "decode_gated" if gated else "decode", "batch": batch, "q_heads": q_heads,
            "kv_heads": kv_heads, "head_dim": head_dim, "dtype": dtype, "rows": 1, "pos0": n_ctx - 1, "top_k": top_k,
            "span_len": span_len, "back": 4 if gated else 2, "fwd": 2 if gated else 0, "window": 1088 if gated else 0,
            "planted": 0}


def listed():
    return [
        # the fp32 path at its benchmark size (configuration 1): one head, checks against exact arithmetic
        _prefill("prefill_f32_4k", 4096, q_heads=1, kv_heads=1, head_dim=64, dtype="f32", top_k=4, span_len=64),
        # a short prompt of odd length, base span length by the paper's rule ceil(sqrt(i)): launches and latency count
        _prefill("prefill_2k_odd", 1999, top_k=4),
        # an ordinary prompt: a quarter of the flagship configuration
        _prefill("prefill_16k", 16384, span_len=128, planted=8),
        # configuration 2, the workload bench.py times
        _prefill("prefill_65k", 65536, span_len=256, planted=16),
        # configuration 3, the largest: two sequences of 262144 tokens, sixteen spans of 1025 tokens a row
        _prefill("prefill_262k_b2", 262144, batch=2, q_heads=16, kv_heads=4, top_k=16, span_len=512),
        # one chunk of a chunked prefill, half way to the context of configuration 4 and with its heads
        _prefill("chunk_4k_at_500k", 4096, pos0=500001, kv_heads=4, top_k=16, span_len=1024),
        # the kernel configuration of the paper: window 1088, two spans, per-span softmax and gate, 32768-token chunks
        dict(_prefill("gated_65k", 65536, top_k=2), kind="gated", back=4, fwd=2, window=1088),
        # a serving step: eight sequences of a few thousand tokens each
        _decode("decode_8k_b8", 8191, batch=8, kv_heads=8, top_k=8),
        # configurations 4 and 5: one sequence of a million and of ten million tokens
        _decode("decode_1m", 1048576, span_len=1024),
        _decode("decode_10m", 10485760, span_len=3072),
        # the paper's kernel configuration in decoding: window, two spans, gate
        _decode("decode_gated_100k", 100003, kv_heads=8, top_k=2, gated=True),
        # prefill from and to pinned host buffers, copies included
        dict(_prefill("host_16k", 16384, span_len=128), kind="host"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c = _drawn(rng)
    del c["name"]
    return c


def _drawn(rng):
    kind = rng.choice(["prefill", "prefill", "chunk", "generic", "gated", "decode", "decode", "decode_gated", "host"])
    q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (32, 4), (16, 4), (8, 2), (16, 2), (16, 8)])
    heads = dict(q_heads=q_heads, kv_heads=kv_heads)
    top_k = rng.choice([2, 4, 8, 8, 16, 16])
    if kind == "generic":   # fp32, or bf16 with head_dim 64
        head_dim, dtype = rng.choice([(64, "f32"), (128, "f32"), (64, "bf16")])
        q_heads, kv_heads = rng.choice([(1, 1), (2, 1), (4, 2)])
        rows = _log_int(rng, 1000, 8192)
        return _prefill("", rows, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, dtype=dtype,
                        top_k=rng.choice([2, 4, 8]), span_len=rng.choice([0, math.isqrt(rows)]))
    if kind == "prefill":
        batch = rng.choice([1, 1, 2])
        rows = _log_int(rng, 1000, 131072 // batch)
        planted = rng.choice([0, 4])
        span_len = math.isqrt(rows) if planted else rng.choice([0, math.isqrt(rows)])
        return _prefill("", rows, batch=batch, top_k=top_k, span_len=span_len, planted=planted, **heads)
    if kind == "chunk":
        rows, pos0 = _log_int(rng, 1000, 8192), _log_int(rng, 16384, 1048576)
        return _prefill("", rows, pos0=pos0, top_k=top_k, span_len=rng.choice([0, math.isqrt(pos0)]), **heads)
    if kind == "gated":
        return dict(_prefill("", _log_int(rng, 4096, 98304), top_k=rng.choice([2, 2, 4]), **heads), kind="gated", back=4,
                    fwd=2, window=1088)
    if kind == "host":
        return dict(_prefill("", _log_int(rng, 4096, 32768), top_k=top_k, **heads), kind="host")
    if kind == "decode":
        batch = rng.choice([1, 1, 2, 4, 8, 16])
        head_dim, dtype = rng.choice([(128, "bf16"), (128, "bf16"), (128, "bf16"), (64, "bf16"), (128, "f32")])
        most = 8388608 * 4 // (kv_heads * batch * (2 if dtype == "f32" else 1))   # caches stay below that of decode_10m
        n_ctx = _log_int(rng, 2000, most)
        return _decode("", n_ctx, batch=batch, head_dim=head_dim, dtype=dtype, top_k=top_k,
                       span_len=rng.choice([0, math.isqrt(n_ctx)]), **heads)
    batch = rng.choice([1, 1, 4])
    return _decode("", _log_int(rng, 4000, 1048576 // batch), batch=batch, top_k=rng.choice([2, 2, 4]), gated=True, **heads)


def _params(c):
    mode = sla.SLA_PER_SPAN if c["kind"] in ("gated", "decode_gated") else sla.SLA_UNION
    return sla.make_params(c["top_k"], c["span_len"], back_factor=c["back"], fwd_factor=c["fwd"], window=c["window"],
                           mode=mode, head_dim=c["head_dim"])


def _normal(shape, dtype, gen):
    return torch.empty(shape, dtype=dtype, device=DEV).normal_(generator=gen)


def _on_grid(t):
    """Rounds to multiples of 1/64 in place (exact in fp32 and in bf16: a power of two, then an integer)."""
    return t.mul_(64).round_().mul_(1 / 64)


def _workload(c, seed):
    return synth.Workload("case", "prefill", c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"], c["rows"],
                          c["dtype"], c["span_len"], c["top_k"], planted_spans=c["planted"], seed=seed)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    dt, B, Hq, Hkv, D = DTYPES[c["dtype"]], c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"]
    n_kv, rows = c["pos0"] + c["rows"], c["rows"]
    params = _params(c)
    decode = c["kind"] in ("decode", "decode_gated")
    q_shape = (B, Hq, D) if decode else (B, Hq, rows, D)
    if c["planted"]:
        x = synth.make_prefill(_workload(c, seed), device=DEV)
    else:
        x = {n: _normal(q_shape, dt, gen) for n in ("q_s", "q")}
        x.update({n: _normal((B, Hkv, n_kv, D), dt, gen) for n in ("k", "v")})
    _on_grid(x["q_s"])
    _on_grid(x["k"])
    layout = sla.make_layout(x["q"], x["k"], decode=decode)
    need = sla.sla_workspace_bytes(layout, params, rows, n_kv)
    out_rows = (B, Hq) if decode else (B, Hq, rows)
    if c["kind"] == "host":
        # the program holds pinned host buffers for the inputs and the results
        need += sla.sla_host_staging_bytes(layout, params, rows)
        x = {n: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for n, t in x.items()}
        buf = dict(out=torch.empty(q_shape, dtype=dt, pin_memory=True),
                   lse=torch.empty(out_rows, dtype=torch.float32, pin_memory=True),
                   anchor=torch.empty(out_rows + (c["top_k"],), dtype=torch.int32, pin_memory=True),
                   score=torch.empty(out_rows + (c["top_k"],), dtype=torch.float32, pin_memory=True))
        return dict(c=c, x=x, p=params, h=sla.Handle(0, need), buf=buf)
    chunks = []
    step = synth.PAPER_CHUNK if c["kind"] == "gated" else rows
    out = torch.empty(q_shape, dtype=dt, device=DEV)
    for r0 in range(0, rows, step):
        n = min(step, rows - r0)
        part = out_rows if decode else (B, Hq, n)
        chunks.append(dict(r0=r0, n=n, anchor=torch.empty(part + (c["top_k"],), dtype=torch.int32, device=DEV),
                           score=torch.empty(part + (c["top_k"],), dtype=torch.float32, device=DEV),
                           lse=torch.empty(part, dtype=torch.float32, device=DEV),
                           lse_span=torch.empty(part + (c["top_k"],), dtype=torch.float32, device=DEV)))
    return dict(c=c, x=x, p=params, h=sla.Handle(0, need), out=out, chunks=chunks)


def run(state):
    c, x, p, h = state["c"], state["x"], state["p"], state["h"]
    if c["kind"] == "host":
        b = state["buf"]
        return sla.sla_prefill_host(h, x["q_s"], x["q"], x["k"], x["v"], p, out=b["out"], lse=b["lse"],
                                    anchor=b["anchor"], score=b["score"])
    out, ch = state["out"], state["chunks"]
    if c["kind"] in ("decode", "decode_gated"):
        o = ch[0]
        return sla.sla_decode_step(h, x["q_s"], x["q"], x["k"], x["v"], c["pos0"] + 1, p, out=out, lse=o["lse"],
                                   out_anchor=o["anchor"], out_score=o["score"])
    if c["kind"] == "prefill":
        o, n_kv = ch[0], c["pos0"] + c["rows"]
        sla.sla_span_search(h, x["q_s"], x["k"], p, q_pos0=c["pos0"], Lkv=n_kv, out_anchor=o["anchor"], out_score=o["score"])
        sla.sla_span_attention(h, x["q"], x["k"], x["v"], o["anchor"], p, q_pos0=c["pos0"], Lkv=n_kv, out=out, lse=o["lse"])
        return out, o["lse"], o["anchor"], o["score"]
    results = [out]
    for o in ch:   # gated: chunk by chunk, every chunk against the keys up to its own end
        r0, r1 = o["r0"], o["r0"] + o["n"]
        sla.sla_span_search(h, x["q_s"][:, :, r0:r1], x["k"], p, q_pos0=r0, Lkv=r1, out_anchor=o["anchor"], out_score=o["score"])
        sla.sla_span_attention_gated(h, x["q"][:, :, r0:r1], x["k"], x["v"], o["anchor"], o["score"], p, q_pos0=r0, Lkv=r1,
                                     out=out[:, :, r0:r1], lse=o["lse"], lse_span=o["lse_span"])
        results += [o["lse"], o["lse_span"], o["anchor"], o["score"]]
    return results


def _union_tokens(c, i, draws):
    """Expected number of keys in the union of `draws` spans of position i whose anchors are drawn evenly from the
    candidates (from those inside planted spans where there are enough of them)."""
    n = math.isqrt(i + 1)
    t = i + 1 - (np.arange(1, n + 1, dtype=np.int64)) ** 2
    t = t[t <= i - c["window"]]
    if c["planted"]:
        starts = synth.planted_starts(_workload(c, 1), 0)
        inside = np.zeros(t.size, dtype=bool)
        for s in starts:
            inside |= (t >= s) & (t < s + 2 * c["span_len"])
        if inside.sum() >= c["top_k"]:
            t = t[inside]
    if t.size == 0:
        return float(min(c["window"], i + 1))
    ell = c["span_len"] if c["span_len"] else math.isqrt(max(i - 1, 0)) + (i > 0)
    lo, hi = np.maximum(t - c["back"] * ell, 0), np.minimum(t + c["fwd"] * ell, i)
    if c["window"]:
        hi = np.minimum(hi, i - c["window"])
    # how many candidate spans cover a key: steps up at lo, down after hi
    at = np.concatenate([lo, hi + 1])
    order = np.argsort(at, kind="stable")
    cover = np.cumsum(np.concatenate([np.ones(t.size), -np.ones(t.size)])[order])[:-1]
    width = np.diff(at[order])
    return float((width * (1 - (1 - cover / t.size) ** draws)).sum()) + min(c["window"], i + 1)


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: scores of all candidates, and the products of
    every row with the keys it attends to (each key once)."""
    c = case
    es = 4 if c["dtype"] == "f32" else 2
    B, Hq, Hkv, D, k, rows = c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"], c["top_k"], c["rows"]
    G, n_kv = Hq // Hkv, c["pos0"] + rows
    if c["kind"] in ("decode", "decode_gated"):
        i = n_kv - 1
        cand = max(0, math.isqrt(n_kv) - math.isqrt(c["window"]))
        small = B * Hq * (3 * D * es + 4 + 8 * k)
        tokens = _union_tokens(c, i, k)
        per_row = tokens
        if c["kind"] == "decode_gated":   # the window enters every span's softmax
            per_row = tokens + (k - 1) * min(c["window"], i + 1)
        return {"bytes": B * Hkv * D * es * (cand + 2 * _union_tokens(c, i, k * G)) + small,
                "flops": B * Hq * D * (2 * cand + 4 * per_row)}
    pos = np.linspace(c["pos0"], n_kv - 1, 33).astype(np.int64)
    cand = float(np.mean([max(0, math.isqrt(int(i) + 1) - math.isqrt(c["window"])) for i in pos]))
    tokens = float(np.mean([_union_tokens(c, int(i), k) for i in pos]))
    bytes_ = B * D * es * (3 * Hq * rows + 2 * Hkv * n_kv) + B * Hq * rows * (4 + 8 * k + (4 * k if c["kind"] == "gated" else 0))
    return {"bytes": bytes_, "flops": B * Hq * rows * D * (2 * cand + 4 * tokens)}


def tolerance(case):
    """About four times what the outputs differ by from the same rows computed in fp64; selections and scores are exact."""
    if case["dtype"] == "f32":
        return {"rel": 1.5e-6, "max": 1.2e-5}            # seen: 2.9e-7 and 1.9e-6
    if case["head_dim"] == 128 and case["kind"] in ("prefill", "gated", "host"):
        return {"rel": 9e-3, "max": 0.1}                 # weights rounded to bf16 before P V; seen: 2.2e-3 and 2.5e-2
    return {"rel": 7e-3, "max": 1.6e-2}                  # one rounding of the result to bf16; seen: 1.7e-3 and 3.9e-3
