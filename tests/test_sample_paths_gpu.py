"""Whether a sampling call builds the packed array, seen by what it allocates,
with the oracle's result either way."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs
from test_walk_paths_gpu import packed_bytes, preferential, ring

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph,instances,per,fanout,builds", [
    # one instance: a few very long rows that few edges lead to do not pay for the array
    ("preferential", 1, 200, [5, 5, 5], False), ("preferential", 1, 15000, [5, 5, 5], False),
    ("star", 1, 10, [25, 10], True),
    # several: one layer of a few entries does not, more do
    ("ring", 2, 20, [10], False), ("preferential", 300, 100, [10, 5], True)])
@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree"])
def test_when_the_array_is_built(graph, instances, per, fanout, builds, bias):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    if graph == "star":
        V, r = 1 << 17, np.random.default_rng(3)
        a = np.concatenate([np.stack([np.full(V - 4, h), np.arange(4, V)], 1) for h in range(4)])
        a = np.unique(np.concatenate([a, a[:, ::-1]]), axis=0)
        off = np.zeros(V + 1, dtype=np.uint64)
        off[1:] = np.cumsum(np.bincount(a[:, 0], minlength=V))
        g = inputs.CSRGraph(off, a[:, 1].astype(np.uint32), r.integers(1, 256, size=len(a)).astype(np.uint32))
    else:
        g = ring(1 << 18, 16) if graph == "ring" else preferential(1 << 16, 12)
    seeds, io = inputs.distinct_seeds(np.full(instances, per, dtype=np.uint64), g.V, 4)
    G = csaw.Graph(g.off, g.col, g.w)
    sizes = []
    G.use_torch_allocator(lambda p, n: sizes.append(n))
    r = csaw.sample(G, seeds, io, fanout, bias, 5)
    G.use_own_allocator()
    G.close()
    ref = oracle.sample(g, seeds, io, fanout, bias, 5)
    assert np.array_equal(r.edge_offsets, ref["edge_off"])
    assert np.array_equal(r.src, ref["src"]) and np.array_equal(r.dst, ref["dst"])
    assert (packed_bytes(g) in sizes) == builds
