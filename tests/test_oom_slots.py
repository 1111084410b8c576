"""Partition slots of out-of-memory sampling: rows are read as whole 32-byte
sectors, so a slot holds as many words past its last edge as such a read takes."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs


def test_slot_words_cover_the_last_sector():
    from paper_2009_09103_gb300 import build, csaw
    build.build()
    words = getattr(csaw.lib(), "_ZN4csaw14oom_slot_wordsEm")   # csaw::oom_slot_words(uint64_t)
    words.argtypes, words.restype = [ctypes.c_uint64], ctypes.c_uint64
    for edges in [*range(1, 40), 8192, 12345, (1 << 33) + 5]:
        assert words(edges) >= (edges + 7) // 8 * 8


@pytest.mark.gpu
@pytest.mark.parametrize("rest", range(8))
@pytest.mark.parametrize("bias", ["uniform", "edge_weight", "neighbor_degree"])
def test_short_rows_at_the_end_of_a_slot(rest, bias):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    # rows of 41 edges but the last, which makes the one partition end at `rest` modulo 8
    V = 200
    d = np.full(V, 41)
    d[-1] += (rest - 41 * V) % 8
    rng = np.random.default_rng(rest)
    off = np.zeros(V + 1, dtype=np.uint64)
    off[1:] = np.cumsum(d)
    col = np.concatenate([np.sort(rng.choice(V, size=n, replace=False)) for n in d]).astype(np.uint32)
    g = inputs.CSRGraph(off, col, rng.integers(1, 256, size=len(col)).astype(np.uint32))
    assert len(col) % 8 == rest
    seeds, io = np.array([V - 1, V - 2, V - 1, 5], dtype=np.uint32), np.array([0, 2, 4], dtype=np.uint64)
    for budget in (16 * len(col), 16 * len(col) // 3):   # one partition and a few
        r, _ = csaw.sample_oom(g.off, g.col, g.w, seeds, io, [9, 40], bias, 3, budget_bytes=budget, slots=2)
        ref = oracle.sample(g, seeds, io, [9, 40], bias, 3)
        assert np.array_equal(r.edge_offsets, ref["edge_off"])
        assert np.array_equal(r.src, ref["src"]) and np.array_equal(r.dst, ref["dst"])
