"""Host side of DenseTailCache: what it refuses before anything is enqueued, and what it keeps between calls (no GPU)."""
import types

import pytest
import torch

from paper_2508_15212_b200.cache import DenseTailCache


def bare(batch=2, heads=4, cap=8, dtype=torch.bfloat16):
    """A DenseTailCache on host memory whose library calls are recorded instead of made."""
    c = object.__new__(DenseTailCache)
    c.block, c.n_tail, c.made = None, 0, []
    c.k_tail, c.v_tail = (torch.zeros(batch, heads, cap, 128, dtype=dtype) for _ in range(2))
    c._row, c._row_dtype = torch.Size((batch, heads, 128)), dtype
    c._calls = lambda: types.SimpleNamespace(append=lambda k, v: c.made.append((k, v)))
    return c


@pytest.mark.parametrize("shape", [(2, 4, 64), (2, 3, 128), (1, 4, 128), (2, 4, 1, 128), (4, 128), (128,), (1024,)])
@pytest.mark.parametrize("which", ["k", "v"])
def test_append_refuses_rows_of_another_shape(shape, which):
    c, good, bad = bare(), torch.zeros(2, 4, 128, dtype=torch.bfloat16), torch.zeros(shape, dtype=torch.bfloat16)
    with pytest.raises(RuntimeError):
        c.append(*((bad, good) if which == "k" else (good, bad)))
    assert c.made == [] and c.n_tail == 0


@pytest.mark.parametrize("bad", [dict(dtype=torch.float32), dict(dtype=torch.float16), dict(dtype=torch.bfloat16, device="meta")])
def test_append_refuses_rows_of_another_type_or_device(bad):
    c, good = bare(), torch.zeros(2, 4, 128, dtype=torch.bfloat16)
    with pytest.raises(RuntimeError):
        c.append(good, torch.zeros(2, 4, 128, **bad))
    assert c.made == [] and c.n_tail == 0


def test_append_accepts_a_tokens_rows_without_leading_ones():
    for c, shape in ((bare(), (2, 4, 128)), (bare(batch=1), (4, 128)), (bare(batch=1, heads=1), (128,))):
        c.append(torch.zeros(shape, dtype=torch.bfloat16), torch.zeros(shape, dtype=torch.bfloat16))
        assert len(c.made) == 1 and c.n_tail == 1
    with pytest.raises(IndexError):
        c = bare(cap=1)
        for _ in range(2):
            c.append(torch.zeros(2, 4, 128, dtype=torch.bfloat16), torch.zeros(2, 4, 128, dtype=torch.bfloat16))
