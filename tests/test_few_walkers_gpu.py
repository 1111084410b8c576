"""Few walkers or instances on a graph with long rows, where the array or the
index pays for the sake of the longest row alone: bit-exact against the oracle."""
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


@pytest.fixture(scope="module")
def graph():
    return inputs.rmat_csr(15, 16, 255, 21)


@pytest.mark.parametrize("n", [1, 31, 257])
@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree", "node2vec"])
def test_walks(csaw, graph, n, bias):
    starts = inputs.uniform_vertices(n, graph.V, 2)
    starts[0] = int(np.argmax(np.diff(graph.off)))
    G = csaw.Graph(graph.off, graph.col, graph.w)
    for length in (1, 9, 90):   # streamed at the shortest, not at the longest
        assert np.array_equal(csaw.walk(G, starts, length, bias, 7), oracle.walk(graph, starts, length, bias, 7)), length
    kw = {"teleport": "restart", "teleport_q32": 1 << 29}
    assert np.array_equal(csaw.walk(G, starts, 90, bias, 8, **kw), oracle.walk(graph, starts, 90, bias, 8, **kw))
    G.close()


@pytest.mark.parametrize("counts", [[1], [5, 0, 16], [16] * 16])
@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree"])
def test_layers(csaw, graph, counts, bias):
    seeds, io = inputs.distinct_seeds(np.array(counts, dtype=np.uint64), graph.V, 4)
    G = csaw.Graph(graph.off, graph.col, graph.w)
    r = csaw.layer_sample(G, seeds, io, [8, 8], bias, 17)
    G.close()
    ref = oracle.sample(graph, seeds, io, [8, 8], bias, 17, layer=True)
    assert np.array_equal(r.edge_offsets, ref["edge_off"])
    assert np.array_equal(r.src, ref["src"]) and np.array_equal(r.dst, ref["dst"])
