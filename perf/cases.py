"""Workloads that the library's speed is judged on, and how one pass of each is run.

A case is one unit of one layer: the new tokens' K/V rows are appended to the paged cache, then every new token
attends to its sequence's cache.  Geometries, batch shapes and length distributions are those of the repository's
configurations (``cf_synth``) and of its benchmark, plus a layer shape with 64 query heads of 64 elements over 8 KV
heads, whose layers alternate full and sliding-window attention with sink logits.

``call`` names the entry points a pass goes through:
  step     cf_kv_append + cf_mixed_attention                   (lengths handed over on every call)
  planned  cf_kv_append_planned + cf_mixed_attention_planned   (one plan per iteration, one pass per layer)
  shared   cf_kv_append + cf_mixed_attention_shared            (common prefix pages described)
  host     cf_mixed_step_host + cf_host_steps_flush            (activations in pinned host memory)
  static   cf_decode_attention_static                          (decode without a context or allocations)
"""
import math

import numpy as np
import torch

import paper_2609_27085_b200 as cf

BLOCK = 16
GEOMETRIES = ((8, 2, 64), (32, 8, 128), (64, 8, 128), (8, 2, 128), (64, 8, 64))   # query heads, KV heads, head_dim


def _case(name="", call="step", geometry=(32, 8, 128), fp8=False, window=0, sinks=False, decode=0, mean=0, sigma=0.0, lo=0, hi=0,
          chunks=0, budget=0, prefix=0, prefix_hi=-1, shared=0, lengths=0):
    """decode sequences with contexts of median ``mean`` (lognormal, ``sigma``) clipped to [lo, hi], or uniform on
    [lo, hi] when ``sigma`` is 0; ``budget`` prefill tokens split over ``chunks`` prompts whose cached prefixes are
    uniform on [prefix, prefix_hi]; ``shared``: tokens at the front of every decode context that are the same pages."""
    c = {"name": name} if name else {}
    c.update(call=call, q_heads=geometry[0], kv_heads=geometry[1], head_dim=geometry[2], fp8=fp8, window=window, sinks=sinks,
             decode=decode, mean=mean, sigma=sigma, lo=lo, hi=hi, chunks=chunks, budget=budget, prefix=prefix,
             prefix_hi=max(prefix, prefix_hi), shared=shared, lengths=lengths)
    return c


def listed():
    return [
        # The smallest mixed unit: what a call costs when there is next to nothing to compute.
        _case("tiny_mixed", geometry=(8, 2, 64), decode=4, lo=256, hi=256, chunks=1, budget=128, prefix=128),
        # A lightly loaded node between bursts: a handful of short sequences, one pass per layer; latency decides.
        _case("decode_few", call="planned", geometry=(64, 8, 64), sinks=True, decode=5, lo=200, hi=3000, lengths=1),
        # Chat decode without borrowed prefill: the bandwidth-bound core of a decode node.
        _case("decode_chat", decode=64, lo=1024, hi=8192),
        # Sub-agents forked from one context: the long common prefix is described to the call.
        _case("decode_shared", call="shared", decode=16, lo=8300, hi=10500, shared=8192),
        # The chat mix: 48 decodes with lognormal contexts beside two 512-token chunks over cached prefixes.
        _case("mixed_chat", decode=48, mean=4096, sigma=0.8, lo=128, hi=16384, chunks=2, budget=1024, prefix=6144),
        # One rank of four of the same batch (a quarter of the heads), plan kept for all layers.
        _case("mixed_chat_tp4", call="planned", geometry=(8, 2, 128), decode=48, mean=4096, sigma=0.8, lo=128, hi=16384, chunks=2,
              budget=1024, prefix=6144),
        # The same unit driven from host buffers: activations cross the host link in both directions.
        _case("mixed_chat_host", call="host", decode=48, mean=4096, sigma=0.8, lo=128, hi=16384, chunks=2, budget=1024, prefix=6144),
        # Agentic mix: few decodes with very long contexts beside a 2048-token chunk deep into a long prompt.
        _case("mixed_agentic", decode=16, lo=8192, hi=32768, chunks=1, budget=2048, prefix=26624),
        # 256 short decodes and four small chunks on an fp8 cache (both directions of its quantisation).
        _case("mixed_fp8", geometry=(64, 8, 128), fp8=True, decode=256, mean=1242, sigma=1.0, lo=64, hi=32768, chunks=4, budget=512,
              prefix=0, prefix_hi=8192),
        # A sliding-window layer with sinks: short visible ranges, many rows.
        _case("mixed_window", call="planned", geometry=(64, 8, 64), window=128, sinks=True, decode=64, lo=1024, hi=8192, chunks=2,
              budget=4096, prefix=500, prefix_hi=8000, lengths=2),
        # Prefill alone, ragged: three prompts whose chunks and prefixes are no multiple of anything.
        _case("prefill_ragged", decode=0, chunks=3, budget=5003, prefix=37, prefix_hi=9000, lengths=3),
        # The largest budget of the sweep beside 256 decodes, eight query heads per KV head.
        _case("mixed_sweep_8192", geometry=(64, 8, 128), decode=256, mean=1242, sigma=1.0, lo=64, hi=32768, chunks=4, budget=8192,
              prefix=0, prefix_hi=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        call = rng.choice(("step", "step", "step", "planned", "planned", "shared", "host", "static"))
        geometry = rng.choice(GEOMETRIES)
        what = rng.choice(("decode", "mixed", "mixed", "prefill")) if call in ("step", "planned", "host") else "decode"
        fp8 = geometry[2] == 128 and call in ("step", "planned", "host") and rng.random() < 0.25
        window = rng.choice((0, 0, 0, 128, 4096)) if call != "shared" else 0
        c = _case(call=call, geometry=geometry, fp8=fp8, window=window, sinks=rng.random() < (0.7 if window else 0.15),
                  lengths=rng.randrange(1 << 20))
        if what != "prefill":
            mean = _log_int(rng, 100, 24000)
            shared = 0
            if call == "shared":
                shared = _log_int(rng, 512, 16384) // BLOCK * BLOCK
                mean = shared + _log_int(rng, 16, 4000)
            c.update(decode=_log_int(rng, 2, 256), mean=mean, sigma=rng.choice((0.3, 0.8, 1.0)), lo=max(2, shared + 1, mean // 16),
                     hi=min(32768, 8 * mean) if not shared else mean + 4000, shared=shared)
        if what != "decode":
            chunks = rng.randint(1, 4)
            prefix = rng.choice((0, _log_int(rng, 16, 24576)))
            c.update(chunks=chunks, budget=max(2 * chunks, _log_int(rng, 64, 8192)), prefix=prefix,
                     prefix_hi=rng.choice((prefix, prefix + _log_int(rng, 16, 8192))))
        if _cost(c) <= most:
            return c


def _lengths(c):
    """(context_len, query_len) of the batch: a property of the case, not of a seed.  Prefill chunks come first."""
    rng = np.random.default_rng(1000 + c["lengths"])
    lc, lq = [], []
    for i in range(c["chunks"]):
        new = c["budget"] // c["chunks"] + (1 if i < c["budget"] % c["chunks"] else 0)
        lq.append(new)
        lc.append(new + int(rng.integers(c["prefix"], c["prefix_hi"] + 1)))
    n = c["decode"]
    if n and c["sigma"]:
        ctx = np.clip(np.rint(np.exp(np.log(c["mean"]) + c["sigma"] * rng.standard_normal(n))), c["lo"], c["hi"])
    else:
        ctx = rng.integers(c["lo"], c["hi"] + 1, size=n)
    lc += [int(x) for x in ctx]
    lq += [1] * n
    return np.asarray(lc, dtype=np.int32), np.asarray(lq, dtype=np.int32)


def work(c):
    """Bytes: every visible cached token once (a shared prefix once for all its sequences), q in, out and lse out, the new
    K/V rows in and into the cache, the block-table entries in use.  Flops: 4 D per (query head, visible pair)."""
    lc, lq = _lengths(c)
    W, D, Hq, Hkv = c["window"], c["head_dim"], c["q_heads"], c["kv_heads"]
    tokens = pairs = 0
    for s, (l, n) in enumerate(zip(lc.astype(np.int64), lq.astype(np.int64))):
        rows = np.arange(l - n + 1, l + 1)
        pairs += int((np.minimum(rows, W) if W else rows).sum())
        seen = int(min(l, W + n - 1)) if W else int(l)
        tokens += seen - (c["shared"] if c["shared"] and s > 0 else 0)
    T, elem = int(lq.sum()), 1 if c["fp8"] else 2
    kv = 2 * Hkv * D
    new = T * kv * (2 + elem) if c["call"] != "static" else 0
    lse = 4 * T * Hq if c["call"] != "host" else 0
    return {"bytes": tokens * kv * elem + new + 2 * T * Hq * D * 2 + lse + 4 * (tokens // BLOCK), "flops": 4 * D * Hq * pairs}


def _cost(c):
    w = work(c)
    return w["bytes"] / 6.5e12 + w["flops"] / 1.3e15


def tolerance(c):
    # Probabilities are rounded to bf16 (an fp8 cache: to fp16 in decode) and outputs to bf16.  Measured over these cases and
    # a dozen drawn ones: against fp64 0.0024 (rel) at most, of which the output's own rounding is 0.0017; between two
    # ways of cutting the sums 0.0028, and in single values 0.022 of the output's root mean square.  Four times that.
    return {"rel": 0.011, "max": 0.09}


class _State:
    """A batch in device memory with everything a serving loop keeps for it."""
    plan = None

    def __del__(self):
        if self.plan is not None:
            cf.cf_plan_destroy(self.plan)


_context = None


def _ctx():
    global _context
    if _context is None:
        _context = cf.cf_create(torch.cuda.current_device())
    return _context


def prepare(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    Hq, Hkv, D = c["q_heads"], c["kv_heads"], c["head_dim"]
    lc, lq = _lengths(c)
    T, S = int(lq.sum()), len(lc)
    need = (lc + BLOCK - 1) // BLOCK
    shared_pages = c["shared"] // BLOCK
    blocks = int(need.sum()) - max(0, S - 1) * shared_pages + 64
    # every sequence's pages are dealt from a permutation of the pool
    perm = torch.randperm(blocks, generator=g, device="cuda", dtype=torch.int32).cpu()
    table = torch.full((S, int(need.max())), -1, dtype=torch.int32)
    at = shared_pages
    for s in range(S):
        own = int(need[s]) - shared_pages
        table[s, :shared_pages] = perm[:shared_pages]
        table[s, shared_pages:shared_pages + own] = perm[at:at + own]
        at += own

    def normal(*shape):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=g)

    st = _State()
    st.call, st.lc, st.lq = c["call"], lc, lq
    scales = {}
    if c["fp8"]:
        # a cache whose per-head scales were calibrated on its values: codes span the format's range
        st.k_scale, st.v_scale = (torch.empty(Hkv, dtype=torch.float32, device="cuda").uniform_(0.01, 0.03, generator=g) for _ in range(2))
        scales = dict(kv_dtype=cf.CF_KV_FP8_E4M3, k_scale=st.k_scale, v_scale=st.v_scale)

        def pool(scale):
            codes = torch.empty((blocks, Hkv, BLOCK, D), dtype=torch.uint8, device="cuda")
            for b in range(0, blocks, 4096):
                x = normal(min(4096, blocks - b), Hkv, BLOCK, D).float() / scale.view(1, -1, 1, 1)
                codes[b:b + 4096] = x.clamp_(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
            return codes
        st.k, st.v = pool(st.k_scale), pool(st.v_scale)
    else:
        st.k, st.v = normal(blocks, Hkv, BLOCK, D), normal(blocks, Hkv, BLOCK, D)
    st.sinks = torch.empty(Hq, dtype=torch.float32, device="cuda").normal_(generator=g) if c["sinks"] else None
    st.desc = cf.make_desc(Hq, Hkv, D, BLOCK, blocks, window_size=c["window"], sink_logits=st.sinks, **scales)
    st.table, st.width = table.cuda(), table.shape[1]
    st.q, st.k_new, st.v_new = normal(T, Hq, D), normal(T, Hkv, D), normal(T, Hkv, D)
    st.out = torch.empty(T, Hq, D, dtype=torch.bfloat16, device="cuda")
    st.lse = torch.empty(T, Hq, dtype=torch.float32, device="cuda")
    if c["call"] == "host":
        st.q, st.k_new, st.v_new, st.out = (x.cpu().pin_memory() for x in (st.q, st.k_new, st.v_new, st.out))
    if c["call"] == "shared":
        st.group = np.where(lq == 1, 0, -1).astype(np.int32)
        st.shared_len = np.where(lq == 1, c["shared"], 0).astype(np.int32)
    if c["call"] == "planned":
        st.plan = cf.cf_plan_create(_ctx(), st.desc, lc, lq, st.width)
    return st


def run(st):
    if st.call == "static":
        cf.cf_decode_attention_static(st.desc, st.q, st.k, st.v, st.table, st.width, st.lc, st.out, st.lse)
        return {"out": st.out, "lse": st.lse}
    ctx = _ctx()
    if st.call == "host":
        cf.cf_mixed_step_host(ctx, st.desc, st.q, st.k_new, st.v_new, st.k, st.v, st.table, st.width, st.lc, st.lq, st.out)
        cf.cf_host_steps_flush(ctx)
        return {"out": st.out, "k_cache": st.k, "v_cache": st.v}
    if st.call == "planned":
        cf.cf_kv_append_planned(st.plan, st.k, st.v, st.k_new, st.v_new, st.table)
        cf.cf_mixed_attention_planned(st.plan, st.q, st.k, st.v, st.table, st.out, st.lse)
    else:
        cf.cf_kv_append(ctx, st.desc, st.k, st.v, st.k_new, st.v_new, st.table, st.width, st.lc, st.lq)
        if st.call == "shared":
            cf.cf_mixed_attention_shared(ctx, st.desc, st.q, st.k, st.v, st.table, st.width, st.lc, st.lq, st.group, st.shared_len,
                                         st.out, st.lse)
        else:
            cf.cf_mixed_attention(ctx, st.desc, st.q, st.k, st.v, st.table, st.width, st.lc, st.lq, st.out, st.lse)
    return {"out": st.out, "lse": st.lse, "k_cache": st.k, "v_cache": st.v}
