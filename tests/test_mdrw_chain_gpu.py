"""Frontier sampling with degree sums on both sides of 32 bits, bit-exact
against the oracle (pools on chip: 32-bit sums kept up to date, 64-bit sums
scanned)."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def csaw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw as c
    return c


# 2048 slots of a hub of 2^21 - 1 neighbours sum to just under 2^32, of 2^21 to it
@pytest.mark.parametrize("d", [2**21 - 1, 2**21])
@pytest.mark.parametrize("pool", [2048, 2017, 33])
def test_star(csaw, d, pool):
    off = np.concatenate([[0], d + np.arange(d + 1)]).astype(np.uint64)
    col = np.concatenate([np.arange(1, d + 1), np.zeros(d)]).astype(np.uint32)
    g = inputs.CSRGraph(off, col, np.ones(2 * d, dtype=np.uint32))
    rng = np.random.default_rng(pool)
    pools = np.where(rng.random((5, pool)) < np.array([[1.0], [0.99], [0.5], [0.01], [0.0]]), 0,
                     rng.integers(1, d + 1, (5, pool))).astype(np.uint32)
    G = csaw.Graph(g.off, g.col, g.w)
    src, dst = csaw.mdrw(G, pools, 300, 7)
    G.close()
    rs, rd = oracle.mdrw(g, pools, 300, 7)
    assert np.array_equal(src, rs) and np.array_equal(dst, rd)
