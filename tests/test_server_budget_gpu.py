"""A served request builds an array only in what the budget has left beside
the estimates; otherwise its rows are streamed, with the same result."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bias", ["edge_weight", "node2vec"])
@pytest.mark.parametrize("budget", [2 << 20, 1 << 30])
def test_arrays_within_the_budget(bias, budget):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    g = inputs.rmat_csr(15, 16, 255, 21)   # 0.9 M edges: 8 MB as an array
    starts = inputs.uniform_vertices(4000, g.V, 2)
    G = csaw.Graph(g.off, g.col, g.w)
    sizes = []
    G.use_torch_allocator(lambda p, n: sizes.append(n))
    srv = csaw.Server(G, budget_bytes=budget, slots=2)
    r = srv.poll(srv.submit_walk(starts, 60, bias, 7))
    srv.close()
    G.use_own_allocator()
    G.close()
    assert np.array_equal(r.path, oracle.walk(g, starts, 60, bias, 7))
    array = 4 * len(g.col)
    assert (max(sizes) > array) == (budget > 1 << 29)
