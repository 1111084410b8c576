"""Walks over the packed search array, bit-exact against the oracle: rows at
block and window edges, sums far from a straight line (the search starts from
a straight line), zero weights, and the largest weights that fit."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu

DEGREES = [0, 1, 7, 8, 9, 63, 64, 65, 255, 256, 257, 511, 513, 2047, 4096, 8191, 8193, 20000, 3, 1]


@pytest.fixture(scope="module")
def csaw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw as c
    return c


def rows(weights, seed):
    """20,001 vertices; the first rows have DEGREES, the rest lead back to them."""
    rng = np.random.default_rng(seed)
    V, k = 20001, len(DEGREES)
    cols = [np.sort(rng.choice(V, size=d, replace=False)) for d in DEGREES]
    cols += [np.sort(rng.choice(k, size=2, replace=False)) for _ in range(V - k)]
    off = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.uint64)
    return inputs.CSRGraph(off, np.concatenate(cols).astype(np.uint32), weights(rng, int(off[-1])))


WEIGHTS = {
    "even": lambda rng, n: rng.integers(1, 256, n).astype(np.uint32),
    "zeros": lambda rng, n: (rng.integers(0, 4, n) == 0).astype(np.uint32) * 3,
    "front": lambda rng, n: np.where(np.arange(n) % 4096 < 9, 1 << 20, 1).astype(np.uint32),
    "back": lambda rng, n: np.where(np.arange(n) % 4096 > 4000, 1 << 20, 0).astype(np.uint32),
    "widest": lambda rng, n: rng.integers(2**26 - 9, 2**26, n).astype(np.uint32),
    "too_wide": lambda rng, n: rng.integers(2**26, 2**27, n).astype(np.uint32),
}


def starts_for(g, length):
    """Enough walkers for a plain call to build the array."""
    visited = np.sqrt(g.E / g.V * float(np.diff(g.off).max()))
    n = int((8.0 * g.E + 25e6) / (length * (250 + 0.3 * visited))) + 1
    return np.resize(np.arange(g.V, dtype=np.uint32), n)


@pytest.mark.parametrize("name", WEIGHTS)
@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree"])
def test_rows_and_weights(csaw, name, bias):
    g = rows(WEIGHTS[name], 5)
    starts = starts_for(g, 12)
    ref = oracle.walk(g, starts, 12, bias, 77)
    tele = oracle.walk(g, starts, 12, bias, 78, teleport="jump", teleport_q32=1 << 30)
    G = csaw.Graph(g.off, g.col, g.w)
    for form in ("plain", "build", "kept"):
        if form == "kept":
            G.build_cdf(bias)
        assert np.array_equal(csaw.walk(G, starts, 12, bias, 77, build_cdf=form == "build"), ref), form
        if form != "build":
            got = csaw.walk(G, starts, 12, bias, 78, teleport="jump", teleport_q32=1 << 30)
            assert np.array_equal(got, tele), form
    G.close()


@pytest.mark.parametrize("tele", ["restart", "jump"])
def test_uniform_teleports(csaw, tele):
    g = rows(WEIGHTS["even"], 6)
    starts = np.arange(g.V, dtype=np.uint32)
    G = csaw.Graph(g.off, g.col, g.w)
    got = csaw.walk(G, starts, 33, "uniform", 3, teleport=tele, teleport_q32=1 << 29)
    G.close()
    assert np.array_equal(got, oracle.walk(g, starts, 33, "uniform", 3, teleport=tele, teleport_q32=1 << 29))
