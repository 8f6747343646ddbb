"""The work a program that serves long responses gives this framework, as cases that can be timed and compared.

A case is a dict of plain values:

    kind       "decode"    one token for every sequence of a full cache (every token evicts one)
               "generate"  one request served from the host: prompt, then `tokens` tokens through host buffers
               "prompt"    a prompt compressed into the cache, then the first token
               "ragged"    a batch of prompts of different lengths, then the first token
    call       decode: "step" (whole stack per call), "layers" (one call per layer, as a model's forward pass does),
               "steps" (`evict_interval` tokens in one call)
    layers, batch, q_heads, kv_heads, head_dim, C, R, fusion, dtype, evict_interval, profile     as in the binding
    prompt     prompt length ("ragged": the longest row's; the shortest has about a quarter of it)
    tokens     "generate": tokens decoded after the prompt

Shapes are those of the benchmark's workloads and of the tests, with the ranges around them: caches of 64 to 8192
tokens, windows of 16 to 200, 1 to 64 layers x rows per call at the usual head ratios, prompts of up to 131072 tokens.
"""
from __future__ import annotations

import math

import torch

from paper_2503_00979_b200 import binding

DEV = "cuda:0"


def _case(name, kind, layers, batch, q_heads, kv_heads, head_dim, C, R, fusion, dtype="bf16", call="step", evict_interval=1,
          profile="recompute", prompt=0, tokens=0):
    c = dict(kind=kind, layers=layers, batch=batch, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, C=C, R=R,
             fusion=fusion, dtype=dtype, call=call, evict_interval=evict_interval, profile=profile, prompt=prompt, tokens=tokens)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: the f32 correctness workload, one layer; launch and latency are all there is
        _case("step f32 tiny", "decode", 1, 1, 8, 2, 64, 64, 16, "sum", dtype="f32"),
        # the flagship: one long response on a 32-layer stack in a 2K cache, the whole stack per call
        _case("step 32 layers", "decode", 32, 1, 32, 8, 128, 2000, 32, "max"),
        # the same stack as a model's forward pass drives it: its layers one after the other
        _case("layer calls", "decode", 32, 1, 32, 8, 128, 2000, 32, "max", call="layers"),
        # serving: 32 sequences decode together in 1K caches
        _case("step batch 32", "decode", 32, 32, 32, 8, 128, 1024, 32, "sum"),
        # long responses at batch 8 in 4K caches with the wider window
        _case("step 4K window 64", "decode", 32, 8, 32, 8, 128, 4000, 64, "max"),
        # a window of 200 recent tokens in a 4K budget
        _case("step window 200", "decode", 32, 1, 32, 8, 128, 3896, 200, "sum"),
        # models with 64-wide heads, a small batch
        _case("step head 64", "decode", 16, 4, 32, 8, 64, 1024, 32, "sum"),
        # coarse-grained eviction: one period of eight tokens in one call
        _case("period of 8", "decode", 32, 1, 32, 8, 128, 2000, 32, "max", call="steps", evict_interval=8),
        # a short request in a budget of 600 at a 7:1 head ratio, served from pinned host buffers: the cache fills for
        # the first 40 tokens and evicts for the other 24
        _case("request 7:1", "generate", 28, 1, 28, 4, 128, 570, 30, "sum", prompt=560, tokens=64),
        # an ordinary long-context prompt into a 2K cache, up to the first token
        _case("prompt 6K", "prompt", 32, 1, 32, 8, 128, 2016, 32, "sum", prompt=6144),
        # the longest prompt
        _case("prompt 128K", "prompt", 32, 1, 32, 8, 128, 2016, 32, "sum", prompt=131072),
        # serving: eight prompts of different lengths are admitted together
        _case("ragged batch 8", "ragged", 32, 8, 32, 8, 128, 1024, 32, "max", prompt=3000),
    ]


# what one pass may cost: key rows visited (decode) and prompt rows (prompt phase) of the largest listed cases
_MOST_KEYS = 32 * 32 * 8 * 1056
_MOST_PROMPT = 32 * 8 * 131072
_HEADS = [(32, 8), (32, 8), (28, 4), (16, 2), (16, 16), (64, 8), (24, 8)]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 7 + ["generate", "prompt", "prompt", "ragged"])
    fusion = rng.choice(["sum", "max"])
    hq, hkv = rng.choice(_HEADS)
    R = rng.choice([16, 30, 32, 32, 48, 64, 100, 200, rng.randint(16, 200)])
    C = _log_int(rng, 512, 8192)
    if kind == "decode":
        call = rng.choice(["step", "step", "step", "layers", "layers", "steps"])
        dtype, d = rng.choice([("bf16", 128)] * 5 + [("bf16", 64), ("f32", 64), ("f32", 128)])
        T, profile = 1, "recompute"
        if call == "steps":
            T = rng.choice([2, 4, 8, 16])
        elif R >= 100 and dtype == "bf16" and d == 128 and rng.random() < 0.3:
            profile = "stored"
        if (dtype, d) != ("bf16", 128):     # the f32 mode and narrow heads: shorter windows, smaller caches
            R, C = min(R, 64), _log_int(rng, 64, 2048)
        # rows of keys weighted by what a pass does to them: tokens per call, window rows, element size
        weight = T * max(1.0, R * (hq // hkv) / 128) * (8.0 if dtype == "f32" else 4.0 if d == 64 else 1.0)
        units = max(1, int(_MOST_KEYS / weight / (C + R) / hkv))
        layers = rng.choice([1, 2, 4, 16, 28, 32])
        if call == "layers":
            layers = max(2, layers)
        layers = min(layers, max(2 if call == "layers" else 1, units))
        batch = min(_log_int(rng, 1, 64), max(1, units // layers))
        return _case(None, kind, layers, batch, hq, hkv, d, C, R, fusion, dtype, call, T, profile)
    layers = rng.choice([8, 16, 28, 32])
    if kind == "generate":
        P, R = _log_int(rng, 64, 2048), min(R, 64)
        C = max(64, P + rng.randint(-P // 2, 64) - R)
        return _case(None, kind, layers, rng.choice([1, 1, 2, 4]), hq, hkv, 128, C, R, fusion, prompt=P,
                     tokens=rng.randint(8, 64))
    C = _log_int(rng, 512, 4096)
    if kind == "prompt":
        weight = max(1.0, R * (hq // hkv) / 128)
        P = _log_int(rng, 600, min(131072, _MOST_PROMPT / weight / layers / hkv))
        batch = max(1, min(rng.choice([1, 1, 2, 4]), int(_MOST_PROMPT / weight / layers / hkv / P)))
        return _case(None, kind, layers, batch, hq, hkv, 128, C, R, fusion, prompt=P)
    R = min(R, 256 // (1 << (hq // hkv - 1).bit_length()))      # ragged batches: a window of at most 256 ring rows
    return _case(None, kind, rng.choice([4, 8, 16]), rng.randint(2, 8), hq, hkv, 128, min(C, 2048), R, fusion,
                 prompt=_log_int(rng, 512, 4096))


# ------------------------------------------------------------------------------------------------ inputs
def _keys(gen, shape):
    """Key rows: normal, one row in fifty four times as long (the heavy rows attention concentrates on)."""
    k = torch.randn(shape, generator=gen, device=DEV)
    heavy = torch.rand(shape[:-1], generator=gen, device=DEV) < 0.02
    return k.mul_(torch.where(heavy, 4.0, 1.0).unsqueeze(-1))


def _queries(gen, keys, G, length):
    """Queries [.., Hq, length, d] that look back at earlier keys [.., Hkv, P, d]: half a random key plus noise."""
    L, B, H, P, d = keys.shape
    j = torch.randint(0, P, (L, B, H, G, length), generator=gen, device=DEV)
    rows = torch.gather(keys.unsqueeze(3).expand(L, B, H, G, P, d), 4, j.unsqueeze(-1).expand(L, B, H, G, length, d))
    q = rows.float().mul_(0.5) + torch.randn(rows.shape, generator=gen, device=DEV)
    return q.view(L, B, H * G, length, d)


def _prompt(gen, c, P, window, n_tokens):
    """Prompt keys and values, the window's queries, and the inputs of `n_tokens` decode steps."""
    L, B, H, d, G = c["layers"], c["batch"], c["kv_heads"], c["head_dim"], c["q_heads"] // c["kv_heads"]
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    k = torch.empty((L, B, H, P, d), dtype=dt, device=DEV)
    v = torch.empty_like(k)
    qw = torch.empty((L, B, H * G, window, d), dtype=dt, device=DEV)
    q = torch.empty((n_tokens, L, B, H * G, d), dtype=dt, device=DEV)
    for l in range(L):
        k[l] = _keys(gen, (B, H, P, d))
        v[l] = torch.randn((B, H, P, d), generator=gen, device=DEV)
        ql = _queries(gen, k[l:l + 1], G, window + n_tokens)[0]
        qw[l] = ql[:, :, :window]
        q[:, l] = ql[:, :, window:].permute(2, 0, 1, 3)
    kn = _keys(gen, (n_tokens, L, B, H, d)).to(dt)
    vn = torch.randn((n_tokens, L, B, H, d), generator=gen, device=DEV).to(dt)
    return k, v, qw, q, kn, vn


def _context(c):
    return binding.MorphKV(c["layers"], c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"], c["C"], c["R"], c["fusion"],
                           c["dtype"], evict_interval=c["evict_interval"], profile=c["profile"])


def _cache(c, mk):
    """The cache's bookkeeping as the context holds it: which token sits in which slot (a token's eviction shows here)
    and the window's normalisers.  (Layers lie one behind the other in the workspace: one view for all of them.)"""
    got, G = {}, c["q_heads"] // c["kv_heads"]
    for name in ("pos", "ring_c"):
        first = mk.view(0)[name]
        L, step = c["layers"], first.numel() * first.element_size()
        assert all(mk.view(l)[name].data_ptr() == first.data_ptr() + l * step for l in range(L))
        t = binding._from_ptr(first.data_ptr(), (L, *first.shape), first.dtype, mk.device)
        got[name] = t[..., :G] if name == "ring_c" else t
    return got


def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    mk = _context(c)
    st = {"case": c, "mk": mk, "i": 0}
    if c["kind"] == "decode":
        P = c["C"] + c["R"]
        n = c["evict_interval"] * max(1, 16 // c["evict_interval"])
        k, v, qw, q, kn, vn = _prompt(gen, c, P, c["R"], n)
        mk.prefill(k, v, qw)
        out = torch.empty_like(q[:c["evict_interval"]] if c["call"] == "steps" else q[0])
        st.update(n=n, out=out, cache=_cache(c, mk))
        T = c["evict_interval"]
        if c["call"] == "steps":
            st["inputs"] = [(q[i:i + T], kn[i:i + T], vn[i:i + T]) for i in range(0, n, T)]
        elif c["call"] == "layers":
            st["inputs"] = [[(l, q[i, l], kn[i, l], vn[i, l], out[l]) for l in range(c["layers"])] for i in range(n)]
        else:
            st["inputs"] = [(q[i], kn[i], vn[i]) for i in range(n)]
        return st
    P, Rw = c["prompt"], min(c["R"], c["prompt"])
    st["k"], st["v"], st["qw"], q, kn, vn = _prompt(gen, c, P, Rw, max(1, c["tokens"]))
    if c["kind"] == "generate":
        st["host"] = [t.cpu().pin_memory() for t in (q, kn, vn)]
        st["steps"] = [tuple(t[i] for t in st["host"]) for i in range(c["tokens"])]
        st["out"] = torch.empty(q.shape, dtype=q.dtype, pin_memory=True)
    else:
        st["first"] = (q[0], kn[0], vn[0])
        st["out"] = torch.empty_like(q[0])
    if c["kind"] == "ragged":
        part = torch.rand(c["batch"], generator=gen, device=DEV).tolist()
        st["lens"] = [P] + [max(1, int(P * (0.25 + 0.75 * x))) for x in part[1:]]
    st["cache"] = None
    return st


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    st, c, mk = state, state["case"], state["mk"]
    if c["kind"] == "decode":
        x = st["inputs"][st["i"]]
        st["i"] = (st["i"] + 1) % len(st["inputs"])
        out = st["out"]
        if c["call"] == "layers":
            for l, q, k, v, o in x:
                mk.decode_step_layer(l, q, k, v, o)
        elif c["call"] == "steps":
            mk.decode_steps(x[0], x[1], x[2], out)
        else:
            mk.decode_step(x[0], x[1], x[2], out)
        return {"out": out, **st["cache"]}
    mk.reset()
    if c["kind"] == "ragged":
        mk.prefill_ragged(st["k"], st["v"], st["qw"], st["lens"])
    else:
        mk.prefill(st["k"], st["v"], st["qw"])
    if c["kind"] == "generate":
        out, stream = st["out"], torch.cuda.current_stream()
        for i, (q, k, v) in enumerate(st["steps"]):
            mk.decode_step_host(q, k, v, out[i])
            stream.synchronize()            # the host reads this token's output before it can send the next token
    else:
        out = mk.decode_step(*st["first"], st["out"])
    if st["cache"] is None:
        st["cache"] = _cache(c, mk)
    return {"out": out, **st["cache"]}


# ------------------------------------------------------------------------------------------------ what it is held to
def work(case):
    """Per decode step and unit: K and V of the cached tokens and the new token's tensors once.  Prompt phase: every
    prompt key and the kept values read once, the kept rows written once; the logits of the window rows."""
    c = case
    e = 4 if c["dtype"] == "f32" else 2
    d, G, R, C = c["head_dim"], c["q_heads"] // c["kv_heads"], c["R"], c["C"]
    U = c["layers"] * c["batch"] * c["kv_heads"]

    def step(n, units):
        return units * (2 * n * d + 2 * G * d + 2 * d) * e, units * 4 * n * G * d

    def prompt(P, units):
        Rw = min(R, P)
        n = min(P, C + Rw)
        return units * (P * d + n * d + 2 * n * d + Rw * G * d) * e, units * 2 * P * Rw * G * d

    if c["kind"] == "decode":
        b, f = step(C + R, U)
        return {"bytes": b * c["evict_interval"], "flops": f * c["evict_interval"]}
    if c["kind"] == "ragged":        # the mean row of the draw
        P = c["prompt"] * (1 + (c["batch"] - 1) * 0.625) / c["batch"]
        b, f = prompt(P, U)
        b2, f2 = step(min(P, C + R), U)
        return {"bytes": b + b2, "flops": f + f2}
    b, f = prompt(c["prompt"], U)
    for i in range(max(1, c["tokens"])):
        b2, f2 = step(min(c["prompt"] + i, C + R), U)
        b, f = b + b2, f + f2
    return {"bytes": b, "flops": f}


def tolerance(case):
    """The tensor-core and the CUDA-core kernels, whose sums run in different orders, give outputs 2e-5 to 8e-5 apart on
    these cases, single values by one step of bf16 (at most 2^-7 of the value: the two fall on either side of a rounding
    boundary), and normalisers 1e-7; the f32 mode with its sums split differently 1.3e-7 and 3e-7.  Of the positions a
    few may differ where two tokens' fused scores tie to rounding; in a prompt's selection that shifts the slots between
    the two."""
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.01}
    return {"rel": 3e-4, "max": 0.03, "differ": 0.01}
