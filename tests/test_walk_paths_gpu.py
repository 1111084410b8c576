"""Which way a walk call goes, seen by what it allocates, at the forms where the
node2vec intersection and the packed array can go wrong: the array or the index
is built in the call, and the paths are the oracle's."""
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


def index_bytes(g):
    return 8 * (g.E // 2 + g.V + 1)


def packed_bytes(g):
    chunks = -(-g.E // 8192)
    return 8 * (chunks * (8192 + 512 + 1) + 4 * (chunks * 128 // 3 + 1) + 2 * (g.V + 1))


def walk(csaw, g, starts, length, bias, seed, mult=(1, 1, 1), kept=False, **tele):
    """Whether the call built its index or array; its paths are checked."""
    G = csaw.Graph(g.off, g.col, g.w)
    if kept:
        G.build_cdf("edge_weight")
    sizes = []
    G.use_torch_allocator(lambda p, n: sizes.append(n))
    got = csaw.walk(G, starts, length, bias, seed, mult, **tele)
    G.use_own_allocator()
    G.close()
    assert np.array_equal(got, oracle.walk(g, starts, length, bias, seed, mult=mult, **tele))
    return (index_bytes(g) if bias == "node2vec" else packed_bytes(g)) in sizes


def hub_graph(V, sizes, wlo, whi, loops=False, seed=6):
    """Hubs 0, 1, ... with so many neighbours each, and one another; loops: self loops too."""
    rng = np.random.default_rng(seed)
    k = len(sizes)
    pairs = [(i, j) for i in range(k) for j in range(i)]
    for i, n in enumerate(sizes):
        pairs += [(i, int(x)) for x in k + rng.choice(V - k, size=n, replace=False)]
    a = np.array(pairs)
    a = np.concatenate([a, a[:, ::-1]])
    if loops:
        a = np.concatenate([a, np.stack([np.arange(0, V, 3)] * 2, 1)])
    a = np.unique(a, axis=0)
    off = np.zeros(V + 1, dtype=np.uint64)
    off[1:] = np.cumsum(np.bincount(a[:, 0], minlength=V))
    return inputs.CSRGraph(off, a[:, 1].astype(np.uint32), rng.integers(wlo, whi + 1, size=len(a)).astype(np.uint32))


def beside_a_star(g, leaves=6000):
    """g and, apart from it, a star: its hub makes the rows that walks come to long in the
    mean, so that calls on g's vertices build the index at sizes the oracle is quick at."""
    V, n = g.V, g.E
    off = np.concatenate([g.off, n + np.arange(1, leaves + 1), [n + 2 * leaves]]).astype(np.uint64)
    col = np.concatenate([g.col, np.full(leaves, V + leaves), V + np.arange(leaves)]).astype(np.uint32)
    w = None if g.w is None else np.concatenate([g.w, np.ones(2 * leaves)]).astype(np.uint32)
    return inputs.CSRGraph(off, col, w)


MULTS = [(1, 2, 4), (0, 1, 1), (1, 0, 2), (4, 1, 0), (0, 0, 1), (1, 0, 0), (0, 1, 0), (0, 0, 0)]


@pytest.mark.parametrize("wlo,whi", [(0, 1), (0, 3), (1, 1), (1, 2**28)])
@pytest.mark.parametrize("mult", MULTS)
@pytest.mark.parametrize("loops", [False, True])
def test_node2vec_weights_and_multipliers(csaw, wlo, whi, mult, loops):
    g = hub_graph(900, (700, 260, 40, 8), wlo, whi, loops)
    starts = np.tile(np.arange(g.V, dtype=np.uint32), 16)
    assert walk(csaw, beside_a_star(g), starts, 10, "node2vec", 21, mult)


@pytest.mark.parametrize("tele", ["restart", "jump"])
@pytest.mark.parametrize("mult", [(0, 1, 1), (1, 0, 0), (0, 0, 1)])
def test_node2vec_teleports(csaw, tele, mult):
    g = hub_graph(900, (700, 260, 40, 8), 0, 3, True)
    starts = np.tile(np.arange(g.V, dtype=np.uint32), 16)
    assert walk(csaw, beside_a_star(g), starts, 10, "node2vec", 22, mult, teleport=tele, teleport_q32=1 << 29)


@pytest.mark.parametrize("sizes", [(1, 1), (3, 9), (31, 130), (129, 700)])
@pytest.mark.parametrize("kept", [False, True])
def test_node2vec_small_rows(csaw, sizes, kept):
    g = hub_graph(2 + 2 * max(sizes) + 50, sizes, 1, 255)
    starts = np.resize(np.array([0, 1, 2, 5], dtype=np.uint32), 60000)
    assert walk(csaw, beside_a_star(g), starts, 60, "node2vec", 23, (3, 1, 2), kept)


@pytest.mark.parametrize("edges,weights", [
    ([(0, 1), (1, 0)], [3, 5]), ([(0, 0)], [1]), ([(0, 0), (0, 1), (1, 0), (1, 1), (1, 2)], [3, 5, 1, 2, 2])])
def test_node2vec_tiny_graphs(csaw, edges, weights):
    g = inputs.csr_from_edges(max(max(e) for e in edges) + 1, edges, weights)
    starts = np.resize(np.arange(g.V, dtype=np.uint32), 50000)
    assert walk(csaw, beside_a_star(g), starts, 90, "node2vec", 2, (1, 2, 4))
    unweighted = inputs.CSRGraph(g.off, g.col, None)
    assert walk(csaw, beside_a_star(unweighted), starts, 90, "node2vec", 3, (1, 2, 4))


@pytest.mark.parametrize("bias,n,length,builds", [
    ("edge_weight", 257, 1, False), ("edge_weight", 257, 12, False), ("edge_weight", 257, 90, False),
    ("edge_weight", 8000, 90, True), ("neighbor_degree", 1, 1, False), ("neighbor_degree", 1, 200, True),
    ("neighbor_degree", 31, 90, True), ("node2vec", 31, 1, False), ("node2vec", 31, 90, True)])
def test_few_walkers(csaw, bias, n, length, builds):
    g = inputs.rmat_csr(15, 16, 255, 21)
    starts = inputs.uniform_vertices(n, g.V, 2)
    starts[0] = int(np.argmax(np.diff(g.off)))
    assert walk(csaw, g, starts, length, bias, 7) == builds
    kw = {"teleport": "restart", "teleport_q32": 1 << 29}
    assert walk(csaw, g, starts, length, bias, 8, **kw) == builds


def ring(V, d):
    """Every vertex beside the d / 2 next and the d / 2 before it."""
    a = np.concatenate([np.arange(-(d // 2), 0), np.arange(1, d // 2 + 1)])
    col = np.sort((np.arange(V)[:, None] + a) % V, axis=1).astype(np.uint32).ravel()
    return inputs.CSRGraph((np.arange(V + 1) * d).astype(np.uint64), col,
                           np.random.default_rng(d).integers(1, 256, size=V * d).astype(np.uint32))


@pytest.mark.parametrize("d,V,n,length", [(4, 1 << 18, 16, 80), (4, 1 << 18, 8000, 80), (64, 1 << 14, 16, 80),
                                          (64, 1 << 14, 30000, 30), (512, 1 << 12, 100, 80)])
def test_node2vec_streams_regular_rows(csaw, d, V, n, length):
    """Where both lists of a step are alike, streaming one is quicker than the index."""
    g = ring(V, d)
    assert not walk(csaw, g, inputs.uniform_vertices(n, V, 2), length, "node2vec", 9, (1, 2, 4))


@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree"])
@pytest.mark.parametrize("d,V", [(4, 1 << 18), (32, 1 << 15), (64, 1 << 16)])
def test_few_walkers_stream_short_rows(csaw, bias, d, V):
    """A few thousand walkers over short rows do not win the array's construction back."""
    g = ring(V, d)
    assert not walk(csaw, g, inputs.uniform_vertices(2000, V, 2), 80, bias, 9)
    assert walk(csaw, g, inputs.uniform_vertices(60000, V, 2), 80, bias, 9)


@pytest.mark.parametrize("tele", ["restart", "jump"])
@pytest.mark.parametrize("n,length,warps", [(1, 32, False), (1, 33, True), (500, 80, True), (1024, 33, True),
                                            (1025, 33, False)])
def test_uniform_teleports(csaw, tele, n, length, warps):
    """Few and long ones by a warp per walker, which takes walkers by a counter."""
    g = inputs.rmat_csr(12, 4, 1, 5)   # isolated vertices among them: dead ends
    starts = inputs.uniform_vertices(n, g.V, 3)
    G = csaw.Graph(g.off, g.col, None)
    sizes = []
    G.use_torch_allocator(lambda p, k: sizes.append(k))
    import torch
    d = torch.from_numpy(starts.view(np.int32)).cuda()
    kw = {"teleport": tele, "teleport_q32": 1 << 29}
    got = csaw.walk(G, d, length, "uniform", 4, **kw)
    host = csaw.walk(G, starts, length, "uniform", 4, **kw)
    G.use_own_allocator()
    G.close()
    ref = oracle.walk(g, starts, length, "uniform", 4, **kw)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), ref) and np.array_equal(host, ref)
    assert (sizes[:1] == [8]) == warps


def preferential(V, m):
    """m edges of every vertex, to earlier ones and most of them to the earliest: a few very
    long rows, which few edges lead to, beside rows of about 2 m."""
    r = np.random.default_rng(5)
    t = np.repeat(np.arange(V), m)
    a = np.stack([t, (r.random(V * m) ** 2 * t).astype(np.int64)], 1)
    a = np.concatenate([a, a[:, ::-1]])
    a = np.unique(a[a[:, 0] != a[:, 1]], axis=0)
    off = np.zeros(V + 1, dtype=np.uint64)
    off[1:] = np.cumsum(np.bincount(a[:, 0], minlength=V))
    return inputs.CSRGraph(off, a[:, 1].astype(np.uint32), r.integers(1, 256, size=len(a)).astype(np.uint32))


@pytest.mark.parametrize("n,length,builds", [(300, 40, False), (300, 120, False), (1000, 40, False), (20000, 120, True)])
def test_rows_that_edges_lead_to(csaw, n, length, builds):
    """It is those that a walk stands on that count, not the longest of the graph."""
    g = preferential(1 << 16, 12)
    starts = inputs.uniform_vertices(n, g.V, 2)
    assert walk(csaw, g, starts, length, "edge_weight", 9) == builds
