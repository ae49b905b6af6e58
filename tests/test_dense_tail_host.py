"""Host side of DenseTailCache: what it refuses before anything is enqueued, and that it keeps no address between calls (no
GPU: the library's two entry points are replaced by one that records its arguments)."""
import copy
import ctypes
import pickle
import types

import pytest
import torch

from paper_2508_15212_b200 import binding as B
from paper_2508_15212_b200.cache import DenseTailCache, SparkCache


@pytest.fixture
def made(monkeypatch):
    """The calls that would have reached the library, as (entry point, integers among the arguments)."""
    calls = []

    def entry(name):
        def f(*args):
            calls.append((name, {a.value if isinstance(a, ctypes.c_void_p) else a for a in args
                                 if isinstance(a, (int, ctypes.c_void_p))}))
            return 0
        return f

    monkeypatch.setattr(B, "_lib", types.SimpleNamespace(**{n: entry(n) for n in ("spark_append_dense", "spark_decode_attn_tail")}))
    monkeypatch.setattr(B, "_stream", lambda: 0)
    return calls


def on_the_host(batch=2, heads=4, cap=8, dtype=torch.bfloat16):
    """A DenseTailCache with an empty tail whose buffers lie in host memory."""
    def side(keep):
        c = object.__new__(SparkCache)
        c.params = B.make_params(batch=batch, n_q_heads=heads, n_kv_heads=heads, window=4, keep=keep, dtype=dtype, n_pool_pages=64)
        c.table_blocks, c.block_table = 4, None
        c.pages, c.packed_lens = torch.zeros(4096, dtype=torch.uint8), torch.zeros(batch, dtype=torch.int32)
        c.qnorm = torch.ones(batch, heads, 128)
        c.ws_compress, c.ws_decode = torch.zeros(512, dtype=torch.uint8), torch.zeros(512, dtype=torch.uint8)
        return c

    c = object.__new__(DenseTailCache)
    c.block, c.n_tail, c._short = None, 0, True
    c._row, c._row_dtype = torch.Size((batch, heads, 128)), dtype
    c.prefix, c.tail = side(64), side(128)
    c.k_tail, c.v_tail = (torch.zeros(batch, heads, cap, 128, dtype=dtype) for _ in range(2))
    c._o, c._l = [torch.zeros(batch, heads, 128) for _ in range(2)], [torch.zeros(batch, heads) for _ in range(2)]
    return c


@pytest.mark.parametrize("shape", [(2, 4, 64), (2, 3, 128), (1, 4, 128), (2, 4, 1, 128), (4, 128), (128,), (1024,)])
@pytest.mark.parametrize("which", ["k", "v"])
def test_append_refuses_rows_of_another_shape(made, shape, which):
    c, good, bad = on_the_host(), torch.zeros(2, 4, 128, dtype=torch.bfloat16), torch.zeros(shape, dtype=torch.bfloat16)
    with pytest.raises(RuntimeError):
        c.append(*((bad, good) if which == "k" else (good, bad)))
    assert made == [] and c.n_tail == 0


@pytest.mark.parametrize("bad", [dict(dtype=torch.float32), dict(dtype=torch.float16), dict(dtype=torch.bfloat16, device="meta")])
def test_append_refuses_rows_of_another_type_or_device(made, bad):
    c, good = on_the_host(), torch.zeros(2, 4, 128, dtype=torch.bfloat16)
    with pytest.raises(RuntimeError):
        c.append(good, torch.zeros(2, 4, 128, **bad))
    assert made == [] and c.n_tail == 0


def test_append_accepts_a_tokens_rows_without_leading_ones(made):
    for i, (c, shape) in enumerate(((on_the_host(), (2, 4, 128)), (on_the_host(batch=1), (4, 128)), (on_the_host(batch=1, heads=1), (128,)))):
        c.append(torch.zeros(shape, dtype=torch.bfloat16), torch.zeros(shape, dtype=torch.bfloat16))
        assert len(made) == i + 1 and c.n_tail == 1
    with pytest.raises(IndexError):
        c = on_the_host(cap=1)
        for _ in range(2):
            c.append(torch.zeros(2, 4, 128, dtype=torch.bfloat16), torch.zeros(2, 4, 128, dtype=torch.bfloat16))


BUFFERS = {"spark_append_dense": ["tail.pages", "tail.packed_lens", "tail.ws_compress", "k_tail", "v_tail"],
           "spark_decode_attn_tail": ["prefix.pages", "prefix.packed_lens", "prefix.qnorm", "prefix.ws_decode", "tail.packed_lens",
                                      "k_tail", "v_tail"]}


@pytest.mark.parametrize("how", ["data", "set_", "object"])
@pytest.mark.parametrize("entry,where", [(e, w) for e, ws in BUFFERS.items() for w in ws])
def test_a_call_takes_the_buffers_as_they_lie_now(made, entry, where, how):
    c, row, q = on_the_host(), torch.zeros(2, 4, 128, dtype=torch.bfloat16), torch.zeros(2, 4, 128, dtype=torch.bfloat16)

    def call():
        if entry == "spark_append_dense":
            c.append(row, row)
        else:
            c.decode(q)
        assert made[-1][0] == entry
        return made[-1][1]

    owner, name = (getattr(c, where.split(".")[0]), where.split(".")[1]) if "." in where else (c, where)
    t = getattr(owner, name)
    old, new, kept = t.data_ptr(), t.clone(), t.detach()      # (kept: the old memory is not handed out again)
    assert old in call()
    if how == "data":
        t.data = new
    elif how == "set_":
        t.set_(new)
    else:
        setattr(owner, name, new)
    args = call()
    assert getattr(owner, name).data_ptr() in args and new.data_ptr() in args and kept.data_ptr() not in args


def test_a_used_cache_can_be_copied_and_stored(made):
    c, row = on_the_host(), torch.zeros(2, 4, 128, dtype=torch.bfloat16)
    c.append(row, row)
    c.decode(row)
    for d in (copy.deepcopy(c), pickle.loads(pickle.dumps(c))):
        assert d.n_tail == 1 and d.k_tail.data_ptr() != c.k_tail.data_ptr()
        d.append(row, row)
        assert {d.k_tail.data_ptr(), d.tail.pages.data_ptr()} <= made[-1][1] and c.k_tail.data_ptr() not in made[-1][1]
