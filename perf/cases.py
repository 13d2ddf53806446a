"""Batches by which the library's speed is measured.

A pass is what an engine does in one iteration for one attention layer, through :class:`PagedAttention`: append the new
tokens' K and V to the paged cache (``write``), partition the batch (``plan``) and compute attention (``run``); its
outputs are the attention output and the log-sum-exps.  One kind of case appends a sequence's tokens and reads the
sequence back instead (``write`` and ``gather``), as an engine does that hands a request's cache on.

A case holds the law of the batch, not its lengths: ``lengths(case)`` draws them from the case's own ``len_seed``.  The
head shapes, page size, length laws and chunk sizes are those of the repository's configurations, tests and sweep:
4/2/64, 32/8/128, 64/8/128 and 8/8/64 heads, 16-token pages, bf16 N(0,1) data, decode contexts uniform around a mean or
lognormal (median 1024, clipped to [16, 16384]), chunks of 2 to 8192 tokens on priors up to 30000.  ``q_scale`` above 1
makes the softmax as peaked as trained heads make it (scores of that standard deviation), so that the running maximum moves.
"""
import math

import numpy as np
import torch

from paper_2507_17769_b200 import PagedAttention

PAGE = 16
FILL_TOKENS = 1 << 18  # tokens drawn and written at a time when a cache is filled


def _case(name, kind, heads, kv_heads, dim, **kw):
    c = {"kind": kind, "heads": heads, "kv_heads": kv_heads, "dim": dim, "fp8": False, "rows": 0, "law": "uniform",
         "ctx_lo": 0, "ctx_hi": 0, "chunks": 0, "chunk_lo": 0, "chunk_hi": 0, "prior_lo": 0, "prior_hi": 0, "q_scale": 1.0,
         "len_seed": 1}
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest mixed iteration: four short decode rows and a 32-token chunk, small heads; launches and latency
        _case("mixed_tiny_d64", "attn", 4, 2, 64, rows=4, ctx_lo=17, ctx_hi=100, chunks=1, chunk_lo=32, chunk_hi=32,
              prior_lo=48, prior_hi=48),
        # a lightly loaded instance: eight decode rows of about 512 tokens (the sweep's smallest decode cell); latency
        _case("decode_few", "attn", 32, 8, 128, rows=8, ctx_lo=256, ctx_hi=768, len_seed=2),
        # an ordinary decode iteration of an 8B-class model: 64 requests
        _case("decode_64", "attn", 32, 8, 128, rows=64, ctx_lo=512, ctx_hi=4096, len_seed=3),
        # the same law on the FP8 cache, with more requests, as the smaller cache allows
        _case("decode_fp8", "attn", 32, 8, 128, fp8=True, rows=160, ctx_lo=512, ctx_hi=4096, len_seed=4),
        # a middle cell of the profiling grid: decode rows and a chunk of which neither dominates
        _case("mixed_grid", "attn", 32, 8, 128, rows=32, ctx_lo=1024, ctx_hi=3072, chunks=1, chunk_lo=512, chunk_hi=512,
              prior_lo=1024, prior_hi=3072, len_seed=5, q_scale=2.0),
        # a full 2048-token budget: 512 decode rows with lognormal contexts and a 1536-token chunk
        _case("mixed_budget", "attn", 32, 8, 128, rows=512, law="lognormal", chunks=1, chunk_lo=1536, chunk_hi=1536,
              prior_lo=0, prior_hi=8192, len_seed=6),
        # four ragged fresh prompts, no prior context: every item is short and causal
        _case("prefill_fresh", "attn", 32, 8, 128, chunks=4, chunk_lo=300, chunk_hi=2050, len_seed=7),
        # one chunk of a long prompt on its earlier context, scores as peaked as trained heads give
        _case("prefill_long", "attn", 32, 8, 128, chunks=1, chunk_lo=2048, chunk_hi=2048, prior_lo=8192, prior_hi=8192,
              len_seed=8, q_scale=3.0),
        # head dimension 64 without head grouping at ordinary size
        _case("mixed_d64", "attn", 8, 8, 64, rows=48, ctx_lo=256, ctx_hi=2048, chunks=2, chunk_lo=700, chunk_hi=1300,
              prior_lo=500, prior_hi=4000, len_seed=9),
        # the largest: long contexts of a large model, two 2048-token chunks beside 256 decode rows, 19 GB of K/V
        _case("mixed_large", "attn", 64, 8, 128, rows=256, ctx_lo=4096, ctx_hi=32768, chunks=2, chunk_lo=2048, chunk_hi=2048,
              prior_lo=16384, prior_hi=30000, len_seed=10),
        # a prompt's cache appended and read back whole
        _case("cache_append_read", "cache", 32, 8, 128, chunks=1, chunk_lo=6001, chunk_hi=6001, prior_lo=0, prior_hi=0,
              len_seed=11),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    heads, kv_heads, dim = rng.choice([(32, 8, 128), (32, 8, 128), (64, 8, 128), (8, 8, 64), (4, 2, 64)])
    kind = rng.choice(["decode", "decode", "fp8", "mixed", "mixed", "mixed", "prefill", "prefill", "cache"])
    kw = {"len_seed": rng.randrange(1 << 30), "q_scale": rng.choice([1.0, 1.0, 2.0, 3.0])}
    if kind == "fp8":
        heads, kv_heads, dim = rng.choice([(32, 8, 128), (64, 8, 128)])
        kw["fp8"] = True
    if kind in ("decode", "fp8", "mixed"):
        kw["rows"] = _log_int(rng, 1, 512)
        if rng.random() < 0.25:
            kw["law"] = "lognormal"
        else:
            mean = _log_int(rng, 64, min(16384, 4_000_000 // kw["rows"]))
            kw["ctx_lo"], kw["ctx_hi"] = mean - mean // 2, mean + mean // 2
    if kind in ("mixed", "prefill"):
        kw["chunks"] = rng.choice([1, 1, 2, 4])
        hi = _log_int(rng, 2, 2048 if heads * dim > 4096 or kind == "mixed" else 4096)
        kw["chunk_lo"], kw["chunk_hi"] = max(2, hi - hi // 2), hi
        prior = rng.choice([0, _log_int(rng, 16, min(16384, 60_000_000 // (kw["chunks"] * hi)))])
        kw["prior_lo"], kw["prior_hi"] = prior - prior // 2, prior
    if kind == "cache":
        kw["chunks"] = 1
        kw["chunk_lo"] = kw["chunk_hi"] = _log_int(rng, 16, 32768)
        kw["prior_lo"] = kw["prior_hi"] = rng.choice([0, _log_int(rng, 16, 32768)])
        kw["q_scale"] = 1.0
    return _case(None, "cache" if kind == "cache" else "attn", heads, kv_heads, dim, **kw)


def lengths(case):
    """(prior, q_len) of the case's requests: decode rows (one new token each), then chunks."""
    rng = np.random.Generator(np.random.PCG64(case["len_seed"]))
    prior, q_len = [], []
    if case["rows"]:
        if case["law"] == "lognormal":
            ctx = np.clip(np.rint(np.exp(math.log(1024) + rng.standard_normal(case["rows"]))), 16, 16384)
        else:
            ctx = rng.integers(case["ctx_lo"], case["ctx_hi"] + 1, case["rows"])
        prior += [int(c) - 1 for c in ctx]
        q_len += [1] * case["rows"]
    for _ in range(case["chunks"]):
        q_len.append(int(rng.integers(case["chunk_lo"], case["chunk_hi"] + 1)))
        prior.append(int(rng.integers(case["prior_lo"], case["prior_hi"] + 1)))
    return np.array(prior, dtype=np.int32), np.array(q_len, dtype=np.int32)


def prepare(case, seed):
    prior, q_len = lengths(case)
    kv_len = prior + q_len
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    heads, kv_heads, dim = case["heads"], case["kv_heads"], case["dim"]

    # pages: a seeded permutation of a pool with a quarter to spare
    need = (kv_len.astype(np.int64) + PAGE - 1) // PAGE
    total = int(need.sum())
    num_pages = max(total + total // 4, total + 8)
    max_pages = int(need.max())
    perm = torch.randperm(num_pages, generator=gen, device=dev, dtype=torch.int32)
    first = torch.from_numpy(np.concatenate([[0], np.cumsum(need)[:-1]])).to(dev)
    slot = torch.arange(max_pages, device=dev)[None, :]
    used = slot < torch.from_numpy(need).to(dev)[:, None]
    table = torch.where(used, perm[(first[:, None] + slot).clamp_(max=num_pages - 1)], 0).to(torch.int32).contiguous()

    pa = PagedAttention(heads, kv_heads, dim, num_pages, kv_dtype=1 if case["fp8"] else 0)

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=dev, dtype=torch.bfloat16)

    # the context cached by earlier iterations, a group of requests (or a stretch of a long one) at a time
    r, done = 0, 0
    while r < len(prior):
        rows, begin, count, tokens = [], [], [], 0
        while r < len(prior) and tokens < FILL_TOKENS:
            take = min(int(prior[r]) - done, FILL_TOKENS - tokens)
            if take > 0:
                rows.append(r)
                begin.append(done)
                count.append(take)
                tokens += take
                done += take
            if done == int(prior[r]):
                r, done = r + 1, 0
        if rows:
            pa.write(normal(tokens, kv_heads, dim), normal(tokens, kv_heads, dim),
                     table[torch.tensor(rows, device=dev)].contiguous(), begin, count, max_pages=max_pages)

    new = int(q_len.sum())
    q = None
    if case["kind"] == "attn":
        q = (torch.randn((new, heads, dim), generator=gen, device=dev) * case["q_scale"]).to(torch.bfloat16)
    return {"kind": case["kind"], "pa": pa, "table": table, "prior": prior, "q_len": q_len, "max_pages": max_pages, "q": q,
            "k_new": normal(new, kv_heads, dim), "v_new": normal(new, kv_heads, dim)}


def run(state):
    pa, table = state["pa"], state["table"]
    pa.write(state["k_new"], state["v_new"], table, state["prior"], state["q_len"])
    if state["kind"] == "cache":
        k, v = pa.gather(table[0], int(state["prior"][0] + state["q_len"][0]))
        return {"k": k, "v": v}
    pa.plan(state["prior"], state["q_len"], state["max_pages"])
    out, lse = pa.run(state["q"], table)
    return {"out": out, "lse": lse}


def work(case):
    prior, q_len = (x.astype(np.float64) for x in lengths(case))
    heads, kv_heads, dim = case["heads"], case["kv_heads"], case["dim"]
    kv_len, new = prior + q_len, q_len.sum()
    token_in = 2 * kv_heads * dim * 2                                            # K and V of a new token, bf16
    token_kv = 2 * kv_heads * (dim + 4) if case["fp8"] else 2 * kv_heads * dim * 2  # K and V of a cached token
    table_bytes = 4 * np.ceil(kv_len / PAGE).sum()
    if case["kind"] == "cache":
        # new tokens read and stored, the earlier ones read, the whole sequence written out
        return {"bytes": float(new * token_in * 2 + prior.sum() * token_kv + kv_len.sum() * token_kv + table_bytes), "flops": 0.0}
    pairs = (q_len * prior + q_len * (q_len + 1) / 2).sum()                      # (new token, visible key) pairs
    return {"bytes": float(new * (token_in + token_kv) + prior.sum() * token_kv + table_bytes + new * heads * (dim * 4 + 4)),
            "flops": float(4.0 * dim * heads * pairs)}


def tolerance(case):
    if case["kind"] == "cache":
        return "exact"
    # About four times what the path shows against the same attention in 64 bits over the cached values: the output's
    # rounding to bf16 (1.66e-3 by itself) and, on the bf16 cache, the softmax weights' (2.0e-3 to 2.3e-3 together; largest
    # single difference 0.033 of the root mean square, in rows with few keys); the FP8 cache's weights are f16.
    return {"rel": 7e-3, "max": 0.02} if case["fp8"] else {"rel": 9e-3, "max": 0.13}
