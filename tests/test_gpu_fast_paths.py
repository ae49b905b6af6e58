"""The selection searches, the division of a decode step among CTAs and the eviction's select kernel at the sizes where
they change branch, against the oracle with the bars of test_gpu_parity.py."""
import ctypes
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_2508_15212_b200 import binding as B
from paper_2508_15212_b200.cache import SparkCache
from test_gpu_parity import built, check_case, check_eviction_case, make, to_np  # noqa: F401  (built: module fixture)

pytestmark = pytest.mark.gpu

LENS = [1, 15, 16, 17, 63]


def tied_workload(kind, seed):
    """Saliencies with many exact ties ("equal"), or distinct ones that share their upper 16 bits ("near")."""
    wl = make("bf16", len(LENS), 8, 2, LENS, 8, 64, seed=seed, gap=False)
    g = torch.Generator(device="cuda").manual_seed(seed)
    sign = torch.where(torch.rand(wl.k.shape, generator=g, device="cuda") < 0.5, -1.0, 1.0)
    if kind == "equal":
        wl.q_win = torch.full_like(wl.q_win, 2.0)
        wl.q_win[..., ::3] = 1.0
        wl.k = (sign * 2.0 ** torch.randint(-1, 2, wl.k.shape, generator=g, device="cuda")).to(wl.k.dtype)
        wl.k[2] = 0.0                                            # a sequence of all-zero keys
    else:
        wl.q_win = (1.0 + 2.0 ** -7 * torch.randint(0, 3, wl.q_win.shape, generator=g, device="cuda")).to(wl.q_win.dtype)
        wl.k = sign.to(wl.k.dtype)
    wl.v = (torch.randint(-2, 3, wl.v.shape, generator=g, device="cuda")).to(wl.v.dtype)
    return wl


@pytest.mark.parametrize("kind", ["equal", "near"])
@pytest.mark.parametrize("keep,keep_v", [(1, 0), (25, 127), (64, 64), (127, 1), (128, 100)])
def test_fixed_selection_with_ties(kind, keep, keep_v):
    check_case(tied_workload(kind, 200 + keep), keep, keep_v=keep_v)


@pytest.mark.parametrize("kind", ["equal", "near"])
@pytest.mark.parametrize("p,cap", [(0.01, 128), (0.5, 128), (0.95, 128), (1.0, 128), (0.95, 40)])
def test_top_p_selection_with_ties(kind, p, cap):
    """Exact sums (few distinct powers of two) or sums far from the goal: the kept sets must be the oracle's."""
    wl = tied_workload(kind, 300)
    wl_cpu = wl.to("cpu")
    _, a = oracle.window_mean(wl_cpu.q_win, 2)
    ref = oracle.select_variant(wl_cpu.k, wl_cpu.seq_lens, a, top_p=p, cap=cap)
    cache = SparkCache(batch=len(LENS), n_q_heads=8, n_kv_heads=2, window=8, keep=cap, dtype="bf16", max_tokens=max(LENS), top_p=p,
                       guard=True)
    cache.compress(wl.q_win, wl.k, wl.v, wl.seq_lens)
    u = cache.unpack(want_v=False)
    assert cache.status() == 0 and cache.broken_guards() == []
    assert np.array_equal(u["mask"].cpu().numpy().view(np.uint32), ref["mask"])
    assert np.allclose(u["mu"].cpu().numpy(), ref["mu"], rtol=1e-6, atol=0)


@pytest.mark.parametrize("close", [1, 2, 7, 8, 9, 16, 128])
@pytest.mark.parametrize("keep,keep_v", [(1, 0), (30, 4), (64, 0), (126, 127)])
def test_fixed_threshold_among_close_keys(close, keep, keep_v):
    """The T-th key lies among `close` keys (and values) that share their upper 16 bits: up to eight are ranked against each
    other, more are admitted value by value or by the descent."""
    lens = [1, 15, 16, 17, 33]
    wl = make("bf16", len(lens), 8, 2, lens, 8, 64, seed=330, gap=False)
    g = torch.Generator(device="cuda").manual_seed(330 + close)
    wl.q_win = (1.0 + 2.0 ** -7 * torch.randint(0, 3, wl.q_win.shape, generator=g, device="cuda")).to(wl.q_win.dtype)
    # octaves by rank, the close keys around rank T; at most 4, so that scores stay below some 50 and the bar of 1e-3 on the
    # log-sum-exp is 300 roundings of them (50 * 2^-24 each)
    for x in (wl.k, wl.v):
        order = torch.rand(x.shape, generator=g, device="cuda").argsort(-1)
        rank = order.argsort(-1).float()
        first = max(0, min(128 - close, keep - close // 2))
        x.copy_(torch.where((rank >= first) & (rank < first + close), 1.0, 2.0 ** ((first - rank) / 8).clamp(-12, 2).round()))
    check_case(wl, keep, keep_v=keep_v)


@pytest.mark.parametrize("close", [1, 7, 8, 9, 60])
@pytest.mark.parametrize("cap", [128, 30])
def test_top_p_threshold_among_close_keys(close, cap):
    """The threshold falls among `close` keys that share their upper 16 bits (up to eight are ranked against each other, more
    go to the rank sort); lengths end in either half of a page.  Few exponents: every sum is exact, the sets are the oracle's."""
    lens = [1, 7, 8, 9, 16, 24, 25, 33]
    wl = make("bf16", len(lens), 8, 2, lens, 8, 64, seed=320, gap=False)
    g = torch.Generator(device="cuda").manual_seed(320 + close)
    wl.q_win = (1.0 + 2.0 ** -7 * torch.randint(0, 3, wl.q_win.shape, generator=g, device="cuda")).to(wl.q_win.dtype)
    k = 2.0 ** torch.randint(-6, -2, wl.k.shape, generator=g, device="cuda").float()
    order = torch.rand(wl.k.shape, generator=g, device="cuda").argsort(-1)
    k.scatter_(-1, order[..., :close], 1.0)
    k.scatter_(-1, order[..., close:close + 3], 4.0)
    wl.k = k.to(wl.k.dtype)
    # goal: the three large keys and half of the close ones
    mid = float((12.0 + 0.5 * close) / k.sum(-1).mean())
    wl_cpu = wl.to("cpu")
    _, a = oracle.window_mean(wl_cpu.q_win, 2)
    ref = oracle.select_variant(wl_cpu.k, wl_cpu.seq_lens, a, top_p=mid, cap=cap)
    cache = SparkCache(batch=len(lens), n_q_heads=8, n_kv_heads=2, window=8, keep=cap, dtype="bf16", max_tokens=max(lens), top_p=mid,
                       guard=True)
    cache.compress(wl.q_win, wl.k, wl.v, wl.seq_lens)
    u = cache.unpack()
    assert cache.status() == 0 and cache.broken_guards() == []
    assert np.array_equal(u["mask"].cpu().numpy().view(np.uint32), ref["mask"])
    assert np.allclose(u["mu"].cpu().numpy(), ref["mu"], rtol=1e-6, atol=0)


@pytest.mark.parametrize("n_seq,longest", [(1, 8200), (2, 8200), (4, 9000), (8, 8500), (9, 8300), (20, 700)])
def test_eviction_select_clusters(n_seq, longest):
    """Eight, four, two and one CTA per (sequence, KV head), by the number of units and the longest prefix."""
    lens = [max(40, longest - 977 * (i % 8)) for i in range(n_seq)]
    check_eviction_case("bf16", lens, 4, 300, 1, Hkv=8, pool=7, seed=501)


@pytest.mark.parametrize("G,W", [(1, 16), (2, 24), (4, 32), (5, 32), (7, 32), (8, 32)])
def test_eviction_votes_at_tile_edges(G, W):
    """One and two blocks of 128 query rows, rows that end inside a block; sequences that end on, before and behind a tile of
    128 keys, in their CTA's first tile or a later one."""
    check_eviction_case("bf16", [127, 128, 129, 255, 256, 257, 1152, 1281, 40], W, 60, G, Hkv=2, pool=3, seed=510 + G)


@pytest.mark.parametrize("G", [4, 5])
def test_eviction_votes_over_many_tiles(G):
    """Up to twenty tiles a CTA with one and two blocks of query rows: every barrier comes back to its first parity and every key
    buffer is used several times; lengths on, before and inside a tile."""
    check_eviction_case("bf16", [5000, 4993, 5120, 5119, 4097, 3000, 5001, 2561], 32, 200, G, Hkv=8, pool=7, seed=525)


@pytest.mark.parametrize("layout", ["token-major", "keys shared by the heads", "keys shared by the sequences", "no more rows than tokens"])
def test_eviction_key_layouts(layout):
    """Every order and stride of the keys that the call takes gives what the same keys in a plain tensor give, also in a cache made
    for longer prompts than it is given."""
    lens = [1000, 1000, 1000] if layout == "no more rows than tokens" else [1000, 130, 640]
    wl = make("bf16", 3, 8, 2, lens, 32, 64, seed=521, gap=False)
    k, v = wl.k, wl.v
    if layout == "token-major":
        k2, v2 = (x.transpose(1, 2).contiguous().transpose(1, 2) for x in (k, v))
    elif layout == "keys shared by the heads":
        k2, v2 = (x[:, :1].expand(-1, 2, -1, -1) for x in (k, v))
    elif layout == "keys shared by the sequences":
        k2, v2 = (x[:1].expand(3, -1, -1, -1) for x in (k, v))
    else:
        k2, v2 = k[:, :, :1000].contiguous(), v[:, :, :1000].contiguous()
    got = []
    for kk, vv, room in ((k2.contiguous(), v2.contiguous(), max(lens)), (k2, v2, 5000)):
        cache = SparkCache(batch=3, n_q_heads=8, n_kv_heads=2, window=32, keep=64, dtype="bf16", max_tokens=room, token_budget=100, guard=True)
        cache.compress(wl.q_win, kk, vv, wl.seq_lens)
        u = cache.unpack()
        assert cache.status() == 0 and cache.broken_guards() == []
        got.append((cache.kept_tokens.clone(), u["mask"][:, :, :100].clone(), u["v"][:, :, :100].clone()))
    for x, y in zip(*got):
        assert torch.equal(x, y)


@pytest.mark.parametrize("G,W", [(4, 32), (8, 32), (8, 64)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_eviction_with_window_queries_off_a_16_byte_boundary(dtype, G, W):
    """The call asks no alignment of the window queries, which the tensor-core votes need: what an aligned copy gives, but for an
    exchange of two tokens with nearly equal votes."""
    wl = make(dtype, 2, 2 * G, 2, [700, 333], W, 64, seed=530 + G, gap=False)
    moved = torch.empty(wl.q_win.numel() + 1, dtype=wl.q_win.dtype, device="cuda")[1:].view(wl.q_win.shape)
    moved.copy_(wl.q_win)
    assert moved.data_ptr() % 16 and wl.q_win.data_ptr() % 16 == 0
    got = []
    for q_win in (wl.q_win, moved):
        cache = SparkCache(batch=2, n_q_heads=2 * G, n_kv_heads=2, window=W, keep=64, dtype=dtype, max_tokens=700, token_budget=100, guard=True)
        cache.compress(q_win, wl.k, wl.v, wl.seq_lens)
        assert cache.status() == 0 and cache.broken_guards() == []
        got.append((cache.kept_tokens.cpu(), cache.qnorm))
    assert torch.equal(got[0][1], got[1][1])
    for x, y in zip(got[0][0].reshape(-1, 100).tolist(), got[1][0].reshape(-1, 100).tolist()):
        assert y == sorted(y) and len(set(x) & set(y)) >= 99


def test_eviction_of_keys_without_a_tensor_map():
    """A stride that a tensor map cannot hold (2^40 bytes and more; to an empty sequence, so no row lies there): the CUDA-core
    passes, with the kept sets of the tensor-core ones but for an exchange of two tokens with nearly equal votes."""
    wl = make("bf16", 2, 8, 2, [1000, 0], 32, 64, seed=535, gap=False)
    got = []
    for stride_b in (wl.k.stride(0), 1 << 40):
        c = SparkCache(batch=2, n_q_heads=8, n_kv_heads=2, window=32, keep=64, dtype="bf16", max_tokens=1000, token_budget=100, guard=True)
        p = [ctypes.c_void_p(t.data_ptr()) for t in (wl.q_win, wl.k, wl.v, wl.seq_lens, c.pages, c.qnorm, c.packed_lens, c.kept_tokens, c.ws_compress)]
        assert B.lib().spark_compress(ctypes.byref(c.params), p[0], p[1], p[2], stride_b, *wl.k.stride()[1:3], p[3], 1000, p[4], None, c.table_blocks,
                                      *p[5:], c.ws_compress.numel(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        assert c.status() == 0 and c.broken_guards() == [] and c.packed_lens.tolist() == [100, 0]
        got.append(c.kept_tokens.cpu())
    assert torch.equal(got[0][1], got[1][1])
    for x, y in zip(got[0][0].tolist(), got[1][0].tolist()):
        assert y == sorted(y) and len(set(x) & set(y)) >= 99


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("n_seq,Hkv,longest,budget", [(2, 2, 700, 100), (3, 2, 90, 100), (32, 8, 80, 40), (33, 8, 80, 40), (33, 8, 30, 40)])
def test_eviction_window_norm(dtype, n_seq, Hkv, longest, budget):
    """The select kernel's window norm (up to 256 units), and the one of its own launch, with prompts that are evicted and
    batches that are kept whole: bit for bit what a call without eviction writes."""
    lens = [longest - 7 * (i % 3) for i in range(n_seq)]
    wl = make(dtype, n_seq, 4 * Hkv, Hkv, lens, 16, 64, seed=540 + n_seq, gap=False)
    norms = []
    for b in (0, budget):
        cache = SparkCache(batch=n_seq, n_q_heads=4 * Hkv, n_kv_heads=Hkv, window=16, keep=64, dtype=dtype, max_tokens=longest, token_budget=b, guard=True)
        cache.compress(wl.q_win, wl.k, wl.v, wl.seq_lens)
        assert cache.status() == 0 and cache.broken_guards() == []
        norms.append(cache.qnorm)
    assert torch.equal(*norms)


@pytest.mark.parametrize("p,cap", [(0.5, 128), (0.95, 128), (1.0, 128), (1.0, 40), (0.95, 40)])
def test_top_p_of_odd_values_equals_appending_them(p, cap):
    """Infinities, NaN, all-zero rows, saliencies over more than 22 octaves (their sums round, and p = 1 asks for all of
    them) and subnormal ones: the prefill keeps what the append kernels, which sort every token's channels, keep."""
    n = 100
    wl = make("bf16", 1, 8, 2, [n], 8, 64, seed=310, gap=False)
    g = torch.Generator(device="cuda").manual_seed(310)
    k = wl.k.float()

    def anywhere(tokens, value, how_many):
        for t in tokens:
            at = torch.randperm(128, generator=g, device="cuda")[:how_many]
            k[:, :, t, at] = value

    anywhere(range(0, 10), float("nan"), 1)
    anywhere(range(5, 12), float("inf"), 2)
    anywhere(range(12, 16), float("nan"), 60)
    k[:, :, 16] = float("nan")
    k[:, :, 17] = float("-inf")
    k[:, :, 18] = 0.0
    for t in range(20, 60):                                      # 40 to 60 octaves, rounded sums
        k[:, :, t] *= 2.0 ** torch.randint(-30, 31, k[:, :, t].shape, generator=g, device="cuda")
    for t in range(60, 80):
        k[:, :, t] *= 2.0 ** -126
    anywhere(range(70, 90), 0.0, 100)
    wl.k = k.to(torch.bfloat16)
    kw = dict(batch=1, n_q_heads=8, n_kv_heads=2, window=8, keep=cap, dtype="bf16", max_tokens=n, top_p=p)
    whole, grown = SparkCache(**kw), SparkCache(**kw)
    whole.compress(wl.q_win, wl.k, wl.v, wl.seq_lens)
    grown.compress(wl.q_win, wl.k, wl.v, torch.zeros_like(wl.seq_lens))
    grown.append_block(wl.k, wl.v)
    assert whole.status() == 0 and grown.status() == 0
    a, b = whole.unpack(), grown.unpack()
    assert torch.equal(a["mask"], b["mask"]) and torch.equal(a["vals"].view(torch.int16), b["vals"].view(torch.int16))
    assert torch.allclose(a["mu"], b["mu"], rtol=1e-6, atol=0, equal_nan=True)


@pytest.mark.parametrize("name,Hq,Hkv,lens", [
    ("units of at most a step per warp", 8, 4, [240, 1, 0, 17]),
    ("units up to three steps per warp that fill the grid", 16, 8, [60 + 42 * i for i in range(16)]),
    ("one step more than that", 16, 8, [721] + [60 + 42 * i for i in range(15)]),
    ("short ragged units, several per CTA", 8, 4, [4000, 150, 700, 1300, 16, 0, 2900, 333]),
    ("more tiny units than an epoch holds", 16, 8, [1 + (7 * i) % 40 for i in range(60)]),
    ("seven heads per group", 28, 4, [100 + 97 * i for i in range(20)]),
    ("equal units, a share of one step more than even", 16, 8, [4096]),
    ("equal units, some with two CTAs", 8, 4, [800] * 32),
    ("unequal units, two heads a group", 16, 8, [150 + 550 * i for i in range(8)]),
    ("unequal units, one head a group, empty sequences", 4, 4, [0, 3000, 0, 17, 1200, 0]),
    ("more sequences than lanes, two heads a group", 4, 2, [30 * (i % 3) for i in range(39)] + [2500]),
    ("as many units as CTAs, two heads a group", 2, 1, [900 + i for i in range(148)]),
    ("unequal units in whole CTAs", 32, 8, [150 + 550 * i for i in range(8)]),
    ("unequal units in whole CTAs, eight heads a group", 16, 2, [150 + 550 * i for i in range(8)]),
    ("unequal units in whole CTAs, empty sequences, CTAs to spare", 16, 4, [0, 3000, 0, 17, 1200, 0]),
    ("more sequences than lanes, whole CTAs", 8, 2, [30 * (i % 3) for i in range(39)] + [2500]),
    ("as many units as CTAs", 8, 1, [900 + i for i in range(148)]),
    ("shares of less than two of the shortest unit", 16, 4, [700, 2500, 900, 1700]),
])
def test_division_of_the_step(name, Hq, Hkv, lens):
    check_case(make("bf16", len(lens), Hq, Hkv, lens, 8, 64, seed=400 + len(lens), gap=False), 64, check_vals=False)


@pytest.mark.parametrize("Hq,Hkv,n", [(1, 1, 1280), (1, 1, 1312), (1, 1, 7500), (2, 1, 4736), (2, 1, 4737), (4, 2, 3000), (3, 3, 1600)])
def test_fp32_units_of_many_parts(Hq, Hkv, n):
    """One and two heads a group, a unit over up to 148 CTAs: one group of 32 parts at a time and two, whole and partly filled."""
    check_case(make("f32", 1, Hq, Hkv, [n], 8, 64, seed=480 + Hq, sigma=0.5, gap=False), 64, check_vals=False)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("Hq,Hkv,lens", [
    (8, 4, [4000, 150, 700, 1300, 16, 0, 2900, 333]),
    (8, 8, [1000] * 20),
    (28, 4, [100 + 97 * i for i in range(20)]),
    (16, 2, [5000, 1, 5000, 40, 3000, 900]),
    (4, 4, [900, 2500, 40]),
    (8, 1, [330, 20, 1000]),
])
def test_division_of_the_step_with_head_room(dtype, Hq, Hkv, lens):
    """Units per epoch and ring slots follow the lengths: a cache with room for sixteen times the longest sequence gives what
    one without gives, bit for bit (the grid, which follows the capacity too, is full in both)."""
    wl = make(dtype, len(lens), Hq, Hkv, lens, 8, 64, seed=450 + len(lens), sigma=1.0 if dtype == "bf16" else 0.5, gap=False)
    check_case(wl, 64, check_vals=False)
    outs = []
    for room in (1, 16):
        cache = SparkCache(batch=len(lens), n_q_heads=Hq, n_kv_heads=Hkv, window=8, keep=64, dtype=dtype, max_tokens=room * max(lens))
        cache.max_src_tokens = max(lens)
        cache.compress(wl.q_win, wl.k, wl.v, wl.seq_lens)
        outs.append(cache.decode(wl.q))
        assert cache.status() == 0
    assert torch.equal(*outs)


@pytest.mark.parametrize("lens,W,budget,G,pool", [
    ([1500, 900], 8, 8, 4, 7),              # the window alone
    ([5000, 4100], 16, 600, 2, 601),        # pooling wider than the staging tile's halo
    ([9000], 4, 1025, 1, 1),                # no pooling, a share that is not full
    ([300001], 4, 64, 1, 7),                # a share beyond shared memory
])
def test_eviction_select_edges(lens, W, budget, G, pool):
    check_eviction_case("bf16", lens, W, budget, G, Hkv=1 if lens[0] > 100000 else 2, pool=pool, seed=500)


def test_threads_with_different_shared_memory_needs():
    """Prompts of two sizes evicted and pruned by three threads on their own streams: the launches of the larger size must
    not depend on what another thread last asked the driver for (set launch by launch, some six calls in 8000 were refused)."""
    made = []
    for n in (200, 200, 20000):
        wl = make("bf16", 1, 1, 1, [n], 4, 64, seed=600, gap=False)
        cache = SparkCache(batch=1, n_q_heads=1, n_kv_heads=1, window=4, keep=64, dtype="bf16", max_tokens=n, token_budget=64)
        cache.compress(wl.q_win, wl.k, wl.v, wl.seq_lens)
        made.append((wl, cache, torch.cuda.Stream()))
    torch.cuda.synchronize()
    refused, start = [0] * len(made), threading.Barrier(len(made))

    def work(i):
        wl, c, stream = made[i]
        p = [ctypes.c_void_p(t.data_ptr()) for t in (wl.q_win, wl.k, wl.v, wl.seq_lens, c.pages, c.qnorm, c.packed_lens, c.kept_tokens, c.ws_compress)]
        args = (ctypes.byref(c.params), p[0], p[1], p[2], *wl.k.stride()[:3], p[3], wl.k.shape[2], p[4], None, c.table_blocks,
                *p[5:], c.ws_compress.numel(), ctypes.c_void_p(stream.cuda_stream))
        start.wait()
        refused[i] = sum(B.lib().spark_compress(*args) != 0 for _ in range(8000))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(made))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert refused == [0] * len(made)
    assert all(cache.status() == 0 for _, cache, _ in made)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_steps_of_several_shapes_take_turns_on_one_workspace(dtype):
    """A batch that grows and shrinks between steps, units split over CTAs in each: the workspace of the largest serves all."""
    made = []
    for Hq, Hkv, lens in ((16, 8, [3000] * 8), (8, 4, [5000]), (4, 4, [900, 2500, 40]), (7, 1, [4000, 4000])):
        wl = make(dtype, len(lens), Hq, Hkv, lens, 8, 64, seed=470 + len(lens), sigma=1.0 if dtype == "bf16" else 0.5, gap=False)
        cache = SparkCache(batch=len(lens), n_q_heads=Hq, n_kv_heads=Hkv, window=8, keep=64, dtype=dtype, max_tokens=max(lens))
        cache.compress(wl.q_win, wl.k, wl.v, wl.seq_lens)
        made.append((cache, wl.q, cache.decode(wl.q).clone()))
        assert cache.status() == 0
    shared = torch.empty(max(c.ws_decode.numel() for c, _, _ in made), dtype=torch.uint8, device="cuda")
    B.spark_workspace_init(shared)
    for i in (0, 1, 0, 2, 3, 0, 3, 1, 2, 0):
        cache, q, want = made[i]
        cache.ws_decode = shared
        assert torch.equal(cache.decode(q, out=torch.full_like(want, float("nan"))), want)
        assert cache.status() == 0
