"""node2vec walks by list intersection, bit-exact against the oracle where the
form can go wrong: both lists' sides, rows of several groups per slot,
clustered ids, zero and wide weights, zero multipliers, teleports, tiny graphs."""
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


def symmetric(V, pairs, wlo, whi, seed):
    """CSR of undirected pairs (int array [m, 2]), weights uniform in [wlo, whi] per direction."""
    rng = np.random.default_rng(seed)
    a = np.concatenate([pairs, pairs[:, ::-1]]).astype(np.uint64)
    a = a[a[:, 0] != a[:, 1]]
    key = np.unique(a[:, 0] << np.uint64(32) | a[:, 1])
    src, col = (key >> np.uint64(32)).astype(np.int64), (key & np.uint64(0xFFFFFFFF)).astype(np.uint32)
    off = np.zeros(V + 1, dtype=np.uint64)
    off[1:] = np.cumsum(np.bincount(src, minlength=V))
    return inputs.CSRGraph(off, col, rng.integers(wlo, whi + 1, size=len(col)).astype(np.uint32))


def hubs(sizes, V, seed, clustered=False):
    """Hub vertices 0..k-1, each adjacent to `sizes[i]` others (and to every hub)."""
    rng = np.random.default_rng(seed)
    k = len(sizes)
    pairs = [(i, j) for i in range(k) for j in range(i)]
    for i, n in enumerate(sizes):
        leaves = k + (np.arange(n) + 17 * i if clustered else rng.choice(V - k, size=n, replace=False))
        pairs += [(i, int(x)) for x in leaves]
    return np.array(pairs)


def check(csaw, g, starts, length, mult, seed, kept=False, **tele):
    # as many walkers as make the call large enough for this path
    d = np.diff(g.off)
    need = (5.0 * g.E + 2e6) / (length * np.sqrt(g.E / g.V * float(d.max())))
    starts = np.resize(starts, max(len(starts), int(need) + 2)).astype(np.uint32)
    G = csaw.Graph(g.off, g.col, g.w)
    if kept:
        G.build_cdf("edge_weight")
    got = csaw.walk(G, starts, length, "node2vec", seed, mult, **tele)
    G.close()
    assert np.array_equal(got, oracle.walk(g, starts, length, "node2vec", seed, mult=mult, **tele))


@pytest.mark.parametrize("sizes", [(1, 1), (3, 9), (31, 130), (129, 4097), (5000, 300), (4096, 12289), (13000, 26000)])
@pytest.mark.parametrize("clustered", [False, True])
def test_hub_pairs(csaw, sizes, clustered):
    V = 2 + 2 * max(sizes) + 50
    g = symmetric(V, hubs(sizes, V, 3, clustered), 1, 255, 5)
    starts = np.concatenate([np.array([0, 1], dtype=np.uint32), inputs.uniform_vertices(300, V, 4)])
    check(csaw, g, starts, 14, (1, 2, 4), 11)
    check(csaw, g, starts, 14, (3, 1, 2), 12, kept=True)


@pytest.mark.parametrize("wlo,whi", [(0, 1), (0, 3), (1, 1), (1, 2**28)])
@pytest.mark.parametrize("mult", [(1, 2, 4), (0, 1, 1), (1, 0, 2), (4, 1, 0), (0, 0, 1), (1, 0, 0), (0, 1, 0)])
def test_weights_and_multipliers(csaw, wlo, whi, mult):
    V = 900
    g = symmetric(V, hubs((700, 260, 40, 8), V, 6), wlo, whi, 7)
    check(csaw, g, np.arange(V, dtype=np.uint32), 10, mult, 21)


@pytest.mark.parametrize("tele", ["restart", "jump"])
def test_teleports(csaw, tele):
    g = symmetric(2000, hubs((1500, 700, 90), 2000, 8), 0, 9, 9)
    starts = np.arange(2000, dtype=np.uint32)
    check(csaw, g, starts, 20, (1, 2, 4), 31, teleport=tele, teleport_q32=1 << 29)


def test_unweighted_and_tiny(csaw):
    g = inputs.rmat_csr(10, 16, 1, 3)
    check(csaw, inputs.CSRGraph(g.off, g.col, None), np.arange(g.V, dtype=np.uint32), 30, (1, 2, 4), 5)
    check(csaw, inputs.csr_from_edges(2, [(0, 1), (1, 0)], [3, 5]), np.array([0, 1, 0], dtype=np.uint32), 9, (1, 2, 4), 2)
    check(csaw, inputs.csr_from_edges(3, [(0, 0), (0, 1), (1, 0), (1, 1), (1, 2)], [3, 5, 1, 2, 2]),
          np.array([0, 1, 2], dtype=np.uint32), 12, (1, 2, 4), 2)
