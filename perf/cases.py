"""The work that is timed: what a program that keeps its attention cache in this library has it do.

Five kinds of pass, all through the package's public objects:

  decode   one decode step over a packed cache with fixed buffers (`SparkCache.bind_decode`), the call that a
           generation loop makes once per layer and token
  step     a generation step with its append: the new token's key and value enter the cache, then the decode step
  tail     a block of generated tokens over a cache whose appended keys stay dense (`DenseTailCache`): every token
           is appended and decoded, the last append hands the block over to the pruned prefix
  prefill  a prompt (or a batch of prompts) is pruned and packed, optionally evicted first, and the first token is
           decoded from it
  export   a batch of prompts is pruned and packed and read back as logical arrays (masks, means, kept values,
           value rows), as a program does that moves the pruned cache elsewhere or looks at it

Values are Gaussian with log-normal per-channel scales and a few strong key channels, as attention keys and queries
have; the observation window's queries share the decode query's scales.
"""
import math

import torch

from paper_2508_15212_b200 import binding
from paper_2508_15212_b200.cache import DenseTailCache, SparkCache

D = 128
PAGE = 16
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
ESIZE = {"f32": 4, "bf16": 2}

DEFAULTS = dict(dtype="bf16", batch=1, q_heads=32, kv_heads=8, low=32768, high=32768, window=32, ratio=0.5,
                ratio_v=0.0, top_p=0.0, budget=0, paged=False, token_major=False, block=0)


def _case(kind, **kw):
    c = dict(DEFAULTS, kind=kind)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one head, a short fp32 cache; launch and latency are all there is
        _case("decode", name="decode_f32_1k", dtype="f32", q_heads=1, kv_heads=1, low=1024, high=1024),
        # one sequence of 32K tokens, 32 query / 8 KV heads: the benchmark's own shape
        _case("decode", name="decode_32k"),
        # long context, strong pruning, a few sequences: the largest plain decode step
        _case("decode", name="decode_4x128k_r80", batch=4, low=131072, high=131072, window=64, ratio=0.8),
        # many sequences that were evicted to 2048 tokens each
        _case("decode", name="decode_32x2k", batch=32, low=2048, high=2048),
        # a serving batch of unequal lengths in a shared page pool, seven query heads per KV head
        _case("decode", name="decode_paged_16_ragged", batch=16, q_heads=28, kv_heads=4, low=8192, high=131072, paged=True),
        # value channels pruned as well (half of the keys' and half of the values' channels)
        _case("decode", name="decode_32k_values", ratio_v=0.5),
        # a chat server's token: eight conversations of unequal length, append and decode
        _case("step", name="step_chat_8", batch=8, low=150, high=4000, paged=True),
        # sixty-four generated tokens whose keys stay dense until their block is full
        _case("tail", name="tail_block_64", batch=2, low=3000, high=7000, block=64),
        # a long prompt pruned as a whole, then its first token
        _case("prefill", name="prefill_32k"),
        # a 128K prompt evicted to 2048 tokens per head before pruning, then its first token
        _case("prefill", name="prefill_evict_128k", low=131072, high=131072, budget=2048),
        # the adaptive rule: as many channels per token as carry 99 % of its saliency
        _case("prefill", name="prefill_adaptive_8k", low=8192, high=8192, ratio=0.0, top_p=0.99),
        # short prompts in one batch, keys as a projection leaves them (token-major), read back as arrays
        _case("export", name="export_chat_8", batch=8, low=100, high=3000, token_major=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["decode", "step", "tail", "prefill", "export"], [8, 3, 1, 6, 1])[0]
    q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (28, 4), (16, 8), (8, 8)])
    ratio = rng.choice([0.3, 0.5, 0.5, 0.7, 0.8])
    window = rng.choice([16, 32, 32, 64])
    if kind == "decode":
        if rng.random() < 0.15:                              # the fp32 configuration: few heads, short caches
            heads = rng.choice([1, 2, 4])
            n = _log_int(rng, 200, 8000)
            return _case(kind, dtype="f32", q_heads=heads * rng.choice([1, 2, 4]), kv_heads=heads, low=n, high=n, window=window,
                         ratio=ratio, batch=rng.choice([1, 1, 2]))
        batch = rng.choice([1, 1, 2, 4, 8, 16, 32])
        high = min(131072, _log_int(rng, 500, 131072), 524288 // batch)
        low = high if rng.random() < 0.5 else max(64, high // rng.randint(2, 10))
        return _case(kind, batch=batch, q_heads=q_heads, kv_heads=kv_heads, low=low, high=high, window=window, ratio=ratio,
                     ratio_v=rng.choice([0.0, 0.0, 0.0, 0.5]), paged=rng.random() < 0.5)
    if kind == "step":
        high = _log_int(rng, 300, 16000)
        return _case(kind, batch=rng.randint(1, 32), q_heads=q_heads, kv_heads=kv_heads, low=max(16, high // rng.randint(1, 20)),
                     high=high, window=window, ratio=ratio, paged=rng.random() < 0.5)
    if kind == "tail":
        high = _log_int(rng, 500, 16000)
        return _case(kind, batch=rng.randint(1, 8), q_heads=q_heads, kv_heads=kv_heads, low=max(100, high // rng.randint(1, 4)),
                     high=high, window=window, ratio=ratio, block=rng.choice([32, 64]))
    if kind == "export":
        high = _log_int(rng, 200, 6000)
        return _case(kind, batch=rng.randint(1, 12), q_heads=q_heads, kv_heads=kv_heads, low=max(64, high // rng.randint(1, 20)),
                     high=high, window=window, ratio=ratio, token_major=rng.random() < 0.5)
    what = rng.choice(["plain", "plain", "plain", "values", "evict", "evict", "adaptive", "f32"])
    if what == "evict":
        n = _log_int(rng, 4000, 131072)
        return _case(kind, batch=1 if n > 30000 else rng.choice([1, 2, 4]), q_heads=q_heads, kv_heads=kv_heads, low=n, high=n,
                     window=rng.choice([16, 32]), ratio=ratio, budget=rng.choice([1024, 2048]))
    if what == "adaptive":
        n = _log_int(rng, 500, 16000)
        return _case(kind, q_heads=q_heads, kv_heads=kv_heads, low=n, high=n, window=window, ratio=0.0,
                     top_p=rng.choice([0.9, 0.95, 0.99]))
    if what == "f32":
        n = _log_int(rng, 200, 8000)
        return _case(kind, dtype="f32", q_heads=8, kv_heads=rng.choice([1, 2, 8]), low=n, high=n, window=window, ratio=ratio)
    batch = rng.choice([1, 1, 2, 4])
    high = _log_int(rng, 300, 65536 // batch)
    low = high if rng.random() < 0.5 else max(64, high // rng.randint(2, 10))
    return _case(kind, batch=batch, q_heads=q_heads, kv_heads=kv_heads, low=low, high=high, window=window, ratio=ratio,
                 ratio_v=0.5 if what == "values" else 0.0, token_major=rng.random() < 0.5)


def _lens(c):
    """The batch's sequence lengths: spread evenly over [low, high], long and short ones taking turns."""
    n = c["batch"]
    if n == 1:
        return [c["high"]]
    even = [c["low"] + (c["high"] - c["low"]) * i // (n - 1) for i in range(n)]
    return [even[(i * 5) % n] for i in range(n)] if n % 5 else even


def _keep(c):
    return D if c["top_p"] else binding.spark_keep_count(D, c["ratio"])


def _keep_v(c):
    return binding.spark_keep_count(D, c["ratio_v"]) if c["ratio_v"] else 0


def _prompt(c, gen):
    """Window queries, keys, values and lengths of the batch's prompts, on the GPU."""
    B, Hq, Hkv, W, S, tdt = c["batch"], c["q_heads"], c["kv_heads"], c["window"], c["high"], DTYPES[c["dtype"]]
    sigma = 0.5 if c["dtype"] == "f32" else 1.0

    def randn(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    scale_q = (1.0 if c["dtype"] == "f32" else 0.1) * torch.exp(sigma * randn(Hq, D))      # scores spread over a few units
    scale_k = torch.exp(sigma * randn(B, Hkv, D))
    scale_v = torch.exp(sigma * randn(B, Hkv, D))
    strong = torch.rand((B, Hkv, D), generator=gen, device="cuda").argsort(-1)[..., :4]
    scale_k.scatter_(-1, strong, scale_k.gather(-1, strong) * 8.0)
    q_win = randn(B, Hq, W, D) * scale_q[:, None]
    # a channel's mean window query is small only by chance: such columns are moved away from zero
    mean = q_win.view(B, Hkv, Hq // Hkv * W, D).mean(2)
    floor = 0.05 * scale_q.view(Hkv, Hq // Hkv, D).mean(1)
    shift = torch.where(mean.abs() < floor, torch.where(mean < 0, -floor, floor) - mean, torch.zeros_like(mean))
    q_win = q_win + shift.repeat_interleave(Hq // Hkv, 1)[:, :, None]
    shape = (B, S, Hkv, D) if c["token_major"] else (B, Hkv, S, D)
    k, v = (torch.empty(shape, dtype=tdt, device="cuda") for _ in range(2))
    if c["token_major"]:
        k, v = k.transpose(1, 2), v.transpose(1, 2)
    for b in range(B):
        k[b] = (randn(Hkv, S, D) * scale_k[b][:, None]).to(tdt)
        v[b] = (randn(Hkv, S, D) * scale_v[b][:, None]).to(tdt)
    return dict(q_win=q_win.to(tdt), k=k, v=v, lens=torch.tensor(_lens(c), dtype=torch.int32, device="cuda"),
                scale_q=scale_q, scale_k=scale_k, scale_v=scale_v)


def _cache(c, gen, room=0):
    B, Hkv, max_tokens = c["batch"], c["kv_heads"], c["high"] + room
    table = pool = None
    if c["paged"]:                                          # a pool with a few spare pages, handed out in no order
        blocks = -(-max_tokens // PAGE)
        pool = B * Hkv * blocks + 64
        table = torch.randperm(pool, generator=gen, device="cuda")[: B * Hkv * blocks].to(torch.int32).view(B, Hkv, blocks)
    return SparkCache(batch=B, n_q_heads=c["q_heads"], n_kv_heads=Hkv, window=c["window"], keep=_keep(c), dtype=c["dtype"],
                      max_tokens=max_tokens, block_table=table, n_pool_pages=pool, token_budget=c["budget"],
                      keep_v=_keep_v(c), top_p=c["top_p"] or None)


def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, Hq, Hkv, tdt = c["batch"], c["q_heads"], c["kv_heads"], DTYPES[c["dtype"]]
    x = _prompt(c, gen)
    n = max(1, c["block"])
    q, k_new, v_new = ((torch.randn((n, B, h, D), generator=gen, device="cuda") * s).to(tdt)
                       for h, s in ((Hq, x["scale_q"]), (Hkv, x["scale_k"]), (Hkv, x["scale_v"])))
    s = dict(kind=c["kind"], q=q[0], lens=x["lens"])
    if c["kind"] == "tail":
        s["cache"] = DenseTailCache(batch=B, n_q_heads=Hq, n_kv_heads=Hkv, window=c["window"], keep=_keep(c), dtype=c["dtype"],
                                    max_tokens=c["high"] + c["block"], tail_block=c["block"])
        s["cache"].compress(x["q_win"], x["k"], x["v"], x["lens"])
        s.update(q=q, k_new=k_new, v_new=v_new, out=torch.empty((n, B, Hq, D), dtype=torch.float32, device="cuda"))
        return s
    s["cache"] = cache = _cache(c, gen, room=PAGE if c["kind"] == "step" else 0)
    s["out"], s["lse"] = cache.alloc_out(), cache.alloc_lse()
    if c["kind"] in ("prefill", "export"):
        s["prompt"] = (x["q_win"], x["k"], x["v"], x["lens"])
    else:
        cache.compress(x["q_win"], x["k"], x["v"], x["lens"])
    if c["kind"] != "export":
        s["decode"] = cache.bind_decode(s["q"], out=s["out"], lse=s["lse"])
    if c["kind"] == "step":
        s["new"] = (k_new[0], v_new[0])
    return s


def run(state):
    cache, kind = state["cache"], state["kind"]
    if kind == "decode":
        state["decode"]()
        return dict(out=state["out"], lse=state["lse"])
    if kind == "step":
        cache.packed_lens.copy_(state["lens"])              # the conversation as it was before this token
        cache.append(*state["new"])
        state["decode"]()
        return dict(out=state["out"], lse=state["lse"], lens=cache.packed_lens)
    if kind == "tail":
        cache.prefix.packed_lens.copy_(state["lens"])       # the conversation as it was before this block
        for q, k, v, out in zip(state["q"], state["k_new"], state["v_new"], state["out"]):
            cache.append(k, v)
            cache.decode(q, out=out)
        return dict(out=state["out"], lens=cache.prefix.packed_lens, tail=cache.tail.packed_lens)
    cache.compress(*state["prompt"])
    if kind == "export":
        return dict(cache.unpack(), qnorm=cache.qnorm, lens=cache.packed_lens)
    state["decode"]()
    got = dict(out=state["out"], lse=state["lse"], qnorm=cache.qnorm, lens=cache.packed_lens)
    if cache.kept_tokens is not None:
        got["kept_tokens"] = cache.kept_tokens
    return got


def _kept(c):
    """Kept key channels per token; under the adaptive rule the mean that these inputs give."""
    return {0.9: 46, 0.95: 63, 0.99: 95}[c["top_p"]] if c["top_p"] else _keep(c)


def _token_bytes(c):
    """Packed bytes of one token of one KV head: kept values, masks, mean, value row."""
    e = ESIZE[c["dtype"]]
    kv = _keep_v(c)
    return e * _kept(c) + 16 + 4 + (e * kv + 16 if kv else e * D)


def work(case):
    c = dict(DEFAULTS, **case)
    e, B, Hq, Hkv, W = ESIZE[c["dtype"]], c["batch"], c["q_heads"], c["kv_heads"], c["window"]
    lens = _lens(c)
    packed = [min(n, c["budget"]) if c["budget"] else n for n in lens]
    step_io = B * Hq * D * (e + 4)                          # query in, output out
    pages = _token_bytes(c) * Hkv * sum(packed)
    attend = 2.0 * Hq * sum(packed) * (_kept(c) + (_keep_v(c) or D))
    if c["kind"] == "decode":
        return dict(bytes=pages + step_io, flops=attend)
    new = 2 * B * Hkv * D * e                               # a token's key and value
    if c["kind"] == "step":
        return dict(bytes=pages + step_io + new, flops=attend)
    if c["kind"] == "tail":
        n = c["block"]
        dense = (2 * e * D) * Hkv * B * n * (n - 1) // 2    # the block's earlier tokens, read by each of its steps
        return dict(bytes=n * (pages + step_io + new) + dense, flops=n * attend)
    rows = Hkv * D * e
    kv = (rows * sum(lens) + rows * sum(packed)) if c["budget"] else 2 * rows * sum(lens)
    votes = 2.0 * Hq * W * D * sum(lens) if c["budget"] else 0.0
    total = dict(bytes=kv + pages + B * Hq * W * D * e, flops=votes)
    if c["kind"] == "export":                               # the packed cache is written, then its content as arrays
        total["bytes"] += pages
    else:
        total["bytes"] += step_io
        total["flops"] += attend
    return total


def tolerance(case):
    # about four times what the outputs differ by from the same sums in 64 bits (measured over these ranges: relative
    # 4e-6 and largest 7e-5 for bf16 storage, 4e-7 and 3e-6 for fp32 storage)
    tol = {"rel": 2e-6, "max": 2e-5} if case.get("dtype") == "f32" else {"rel": 1.5e-5, "max": 3e-4}
    if case.get("budget"):                                  # an exchange of two tokens with nearly equal votes
        tol["differ"] = 0.01
    return tol
