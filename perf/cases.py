"""The work that is timed: what a serving program asks of the compressed KV cache, through its public entry points.

A case is one call pattern (`call`) over a cache of a given kind and size:

  prefill   encode a prompt into an empty cache (possibly several prompts of different lengths, packed)
  decode    one query per sequence over what is cached
  stream    `steps` generation steps: append one token per sequence, attend
  chunk     encode the next `new` tokens of every sequence, then their `new` queries attend causally
            (a chunk of a long prefill, or the drafted tokens of a speculative step)
  online    cluster the codebooks on a prompt's own angles, then encode the prompt with them
  window    one query per sequence over the compressed cache and an uncompressed window of recent tokens
  general   any recursion depth and bit table: encode the next `new` tokens of every sequence, then attend

Lengths are a property of the case (`spread` says how ragged they are); values come from the seed.
"""
from __future__ import annotations

import functools
import math
import random

import torch

import paper_2502_02617_b200 as pq
from paper_2502_02617_b200 import synthetic

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
PAGE_TOKENS = 256


def _case(call, **kw):
    c = {"call": call, "batch": 1, "context": 0, "spread": 1.0, "new": 0, "steps": 0, "window": 0, "q_heads": 32, "kv_heads": 8,
         "head_dim": 128, "bits": "4,2,2,2", "dtype": "bf16", "paged": False}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call there is: one sequence, one head of 16 coordinates, 256 tokens in float32 (the repository's
        # "tiny reference" configuration), one generation step.
        _case("stream", name="tiny_d16_f32", context=256, steps=1, q_heads=1, kv_heads=1, head_dim=16, dtype="f32"),
        # An interactive session: one user, a short context, token after token.  Launches and host work count.
        _case("stream", name="stream_b1_short", context=700, steps=8),
        # A loaded server's decode step of one layer: eight sequences of 32k tokens, 32 query / 8 kv heads.
        _case("decode", name="decode_b8_32k", batch=8, context=32768),
        # One layer of a long-context decode step: a single sequence of 128k tokens.
        _case("decode", name="decode_b1_128k", batch=1, context=131072),
        # Continuous batching: sixteen sequences between 4k and 64k tokens behind a block table, appending and attending.
        _case("stream", name="stream_b16_ragged_paged", batch=16, context=65536, spread=16.0, steps=4, paged=True),
        # Prefill of one long prompt.
        _case("prefill", name="prefill_32k", context=32768),
        # A chunk of a long prefill in eight sequences, over what they have cached so far.
        _case("chunk", name="chunk64_b8_32k", batch=8, context=32768, new=64),
        # Verification of drafted tokens in four sequences of uneven length.
        _case("chunk", name="draft5_b4_8k", batch=4, context=8192, spread=3.0, new=5),
        # Prefill of a 16k prompt with codebooks clustered on the prompt itself.
        _case("online", name="online_16k", context=16384),
        # The generated tokens are kept in 16 bits: compressed prompt and window attended together.
        _case("window", name="window_b8_16k", batch=8, context=16384, window=1024, spread=2.0),
        # A smaller model's heads.
        _case("stream", name="stream_d64_b8_4k", batch=8, context=4096, spread=2.0, steps=4, q_heads=16, head_dim=64),
        # The full recursion with three bits per angle.
        _case("general", name="general_full_3bit", batch=8, context=4096, new=512, bits="3,3,3,3,3,3,3"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: the same calls, sizes spread over the whole range of each, odd ones included."""
    most = max(_cost(c) for c in listed())
    while True:
        call = rng.choice(["prefill", "decode", "decode", "stream", "stream", "chunk", "chunk", "online", "window", "general"])
        q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (32, 8), (16, 2), (28, 4), (8, 8)])
        spread = rng.choice([1.0, 1.0, round(rng.uniform(1.5, 16.0), 2)])
        paged = rng.random() < 0.3
        dtype = "f32" if rng.random() < 0.2 else "bf16"
        head_dim = rng.choice([128, 128, 128, 128, 128, 128, 64, 64, 32, 16])
        if call == "prefill":
            c = _case(call, batch=_log_int(rng, 1, 8), context=_log_int(rng, 128, 32768), spread=spread, paged=paged, dtype=dtype,
                      head_dim=head_dim)
        elif call == "decode":
            c = _case(call, batch=_log_int(rng, 1, 32), context=_log_int(rng, 256, 131072), spread=spread, paged=paged, dtype=dtype,
                      head_dim=head_dim)
        elif call == "stream":
            c = _case(call, batch=_log_int(rng, 1, 32), context=_log_int(rng, 256, 65536), spread=spread, steps=rng.randint(1, 8),
                      paged=paged, dtype=dtype, head_dim=head_dim)
        elif call == "chunk":
            c = _case(call, batch=_log_int(rng, 1, 8), context=_log_int(rng, 1024, 32768), spread=spread,
                      new=_log_int(rng, 2, 256), paged=paged, dtype=dtype)
        elif call == "online":
            c = _case(call, context=_log_int(rng, 1024, 32768))
        elif call == "window":
            c = _case(call, batch=_log_int(rng, 1, 16), context=_log_int(rng, 512, 32768), spread=spread,
                      window=_log_int(rng, 32, 2048), paged=paged)
        else:
            head_dim, bits = rng.choice([(128, "3,3,3,3,3,3,3"), (64, "4,3,2"), (256, "4,2,2,2,2"), (128, "4,2,2,2")])
            c = _case(call, batch=_log_int(rng, 1, 8), context=_log_int(rng, 300, 8192), spread=spread,
                      new=_log_int(rng, 1, 256), head_dim=head_dim, bits=bits, dtype=dtype)
        c.update(q_heads=q_heads, kv_heads=kv_heads)
        tokens = sum(_lengths(c))
        if c["head_dim"] < 128 and tokens > 65536:   # the smaller heads belong to smaller models
            continue
        if tokens <= 700000 and _cost(c) <= most:
            return c


def _lengths(case):
    """Tokens cached (or, for a prompt, to be encoded) of each sequence: from context / spread to context, uneven."""
    B, top = case["batch"], case["context"]
    low = max(1, case["new"], case["steps"], int(top / case["spread"]))
    if low >= top:
        return [top] * B
    r = random.Random(B * 1000003 + top)
    return [top] + [r.randint(low, top) for _ in range(B - 1)]


def _windows(case):
    B, T = case["batch"], case["window"]
    r = random.Random(B * 7919 + T)
    return [T] + [r.randint(max(1, T // 2), T) for _ in range(B - 1)]


def _packed_bytes(case):
    """Bytes of one compressed vector (one token of one kv head, K or V)."""
    d, bits = case["head_dim"], [int(b) for b in case["bits"].split(",")]
    return sum(-(-((d >> (l + 1)) * b) // 8) for l, b in enumerate(bits)) + 2 * (d >> len(bits))


def work(case):
    d, hq, hkv = case["head_dim"], case["q_heads"], case["kv_heads"]
    size, packed = (4 if case["dtype"] == "f32" else 2), _packed_bytes(case)
    lens = _lengths(case)
    bytes_ = flops = 0.0

    def encode(n_tokens):
        nonlocal bytes_, flops
        bytes_ += 2 * n_tokens * hkv * (d * size + packed)
        flops += 2 * n_tokens * hkv * 2 * d * d

    def attend(n_cached, n_pairs, n_queries):
        """n_pairs: (query, visible token) pairs summed over the sequences."""
        nonlocal bytes_, flops
        bytes_ += 2 * n_cached * hkv * packed + 2 * n_queries * hq * d * size
        flops += 4 * d * hq * n_pairs

    total, B, new = sum(lens), case["batch"], case["new"]
    if case["call"] == "prefill":
        encode(total)
    elif case["call"] == "online":     # the prompt is clustered first, then encoded: it is read in each of the two
        encode(total)
        bytes_ += 2 * total * hkv * d * size
        flops += 2 * total * hkv * 2 * d * d
    elif case["call"] == "decode":
        attend(total, total, B)
    elif case["call"] == "stream":
        for s in range(case["steps"]):
            encode(B)
            n = total - B * (case["steps"] - 1 - s)
            attend(n, n, B)
    elif case["call"] == "chunk":
        encode(B * new)
        attend(total, sum(n * new - new * (new - 1) / 2 for n in lens), B * new)
    elif case["call"] == "general":
        encode(B * new)
        attend(total, total, B)
    elif case["call"] == "window":
        w = sum(_windows(case))
        attend(total, total + w, B)
        bytes_ += 2 * w * hkv * d * size
    return {"bytes": bytes_, "flops": flops}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def tolerance(case):
    # Codes are decided as in float64.  A block radius is one rounding to fp16 of a norm formed in float32: an equally
    # accurate norm may round to the neighbour for 0.25 % of the radii, which are at most a quarter of a vector's bytes.
    codes = 6e-4
    if case["call"] == "prefill":
        return {"rel": 1e-6, "differ": codes}
    if case["call"] == "online":       # centroids are float64 means of histogram counts of float32 angles
        return {"rel": 1e-5, "differ": codes}
    if case["dtype"] == "bf16":
        return {"rel": 1e-2, "differ": codes}
    # float32 in and out: at head_dim 128 keys and values are decoded in fp16 pairs and values in fp16; elsewhere float32
    f16 = case["call"] in ("decode", "stream", "chunk", "window") and case["head_dim"] == 128
    return {"rel": 2e-3 if f16 else 5e-5, "differ": codes}


@functools.lru_cache(maxsize=None)
def _general_codebooks(head_dim, bits):
    return pq.pq_general_fit_codebooks(pq.GeneralConfig.of(head_dim, bits))


@functools.lru_cache(maxsize=None)
def _codebooks():
    return pq.pq_fit_codebooks()


def _make_cache(case, capacity, seed):
    B, hq, hkv, d = case["batch"], case["q_heads"], case["kv_heads"], case["head_dim"]
    if case["call"] == "general":
        bits = tuple(int(b) for b in case["bits"].split(","))
        cache = pq.GeneralPolarQuantCache(B, hq, hkv, d, bits, capacity, seed=seed, codebooks=_general_codebooks(d, bits))
    elif case["paged"]:
        per_seq = -(-capacity // PAGE_TOKENS)
        table = torch.randperm(B * per_seq, generator=torch.Generator().manual_seed(seed)).view(B, per_seq)
        cache = pq.PagedPolarQuantCache(B, hq, hkv, d, PAGE_TOKENS, B * per_seq, table, seed=seed, codebooks=_codebooks())
    else:
        cache = pq.PolarQuantCache(B, hq, hkv, d, capacity, seed=seed, codebooks=_codebooks())
    cache.cache.zero_()
    return cache


def _cu(lens, device):
    return torch.tensor([0] + [sum(lens[:i + 1]) for i in range(len(lens))], dtype=torch.int32, device=device)


def _rows(seed, n, case, device):
    return synthetic.kv_like(seed, n, case["kv_heads"], case["head_dim"], DTYPES[case["dtype"]], device)


def _fill(cache, case, counts, seed, device):
    """Encode counts[b] tokens into every sequence, in pieces of at most 32768."""
    B = case["batch"]
    for b, n in enumerate(counts):
        done = 0
        while done < n:
            m = min(32768, n - done)
            K, V = _rows(seed + 7 * b + 1000 * done, m, case, device)
            cache.encode(K, V, _cu([m if i == b else 0 for i in range(B)], device))
            done += m


def prepare(case, seed):
    dev, dt = torch.device("cuda"), DTYPES[case["dtype"]]
    B, hq, d, new, steps = case["batch"], case["q_heads"], case["head_dim"], case["new"], case["steps"]
    lens, call = _lengths(case), case["call"]
    cache = _make_cache(case, max(lens), seed)
    s = {"call": call, "cache": cache}
    if call in ("prefill", "online"):
        s["K"], s["V"] = _rows(seed + 1, sum(lens), case, dev)
        s["cu"] = _cu(lens, dev)
        s["start"] = cache.lens.clone()
        return s
    grown = new if call in ("chunk", "general") else steps
    before = [max(0, n - grown) for n in lens]
    _fill(cache, case, before, 31 * seed + 5, dev)
    s["start"] = cache.lens.clone()
    if call in ("chunk", "general"):
        s["K"], s["V"] = _rows(seed + 1, B * new, case, dev)
        s["cu"] = _cu([new] * B, dev)
    if call == "chunk":
        s["q"] = synthetic.queries(seed + 2, B * new, hq, d, dt, dev).view(B, new, hq, d)
    elif call == "stream":
        s["tokens"] = [(_rows(seed + 100 + i, B, case, dev), synthetic.queries(seed + 200 + i, B, hq, d, dt, dev)) for i in range(steps)]
    else:
        s["q"] = synthetic.queries(seed + 2, B, hq, d, dt, dev)
    if call == "window":
        T = case["window"]
        k, v = _rows(seed + 3, B * T, case, dev)
        s["tail"] = tuple(t.view(B, T, case["kv_heads"], d) for t in (k, v)) + (torch.tensor(_windows(case), dtype=torch.int32, device=dev),)
    return s


def run(s):
    cache, call = s["cache"], s["call"]
    if call == "decode":
        return {"out": cache.attend(s["q"])}
    if call == "window":
        return {"out": cache.attend_with_tail(s["q"], *s["tail"])}
    cache.lens.copy_(s["start"])       # a new turn over the same cached prefix (a new prompt: an empty cache)
    if call == "stream":
        outs = []
        for (k, v), q in s["tokens"]:
            cache.append(k, v)
            outs.append(cache.attend(q))
        return {"out": outs, "cache": cache.cache, "lens": cache.lens}
    if call == "online":
        cache.fit_online_codebooks(s["K"], s["V"])
    cache.encode(s["K"], s["V"], s["cu"])
    r = {"cache": cache.cache, "lens": cache.lens}
    if call == "online":
        r["centroids"] = cache.centroids
    elif call == "chunk":
        r["out"] = cache.attend_multi(s["q"])
    elif call == "general":
        r["out"] = cache.attend(s["q"])
    return r
