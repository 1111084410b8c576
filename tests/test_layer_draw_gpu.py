"""Layer sampling by blocks over the packed array, bit-exact against the
oracle at the edges of its rounds, its table and its shared prefix, and where
repeated sampling runs out of attempts."""
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


def check(csaw, g, seeds, io, sizes, bias, cap=None, kept=False):
    G = csaw.Graph(g.off, g.col, g.w)
    if kept:
        G.build_cdf(bias)
    r = csaw.layer_sample(G, seeds, io, sizes, bias, 17, attempt_cap=cap)
    G.close()
    kw = {} if cap is None else {"attempt_cap": cap}
    ref = oracle.sample(g, seeds, io, sizes, bias, 17, layer=True, **kw)
    assert np.array_equal(r.edge_offsets, ref["edge_off"])
    assert np.array_equal(r.frontier_sizes, ref["fsize"][:len(r.frontier_sizes)])
    assert np.array_equal(r.src, ref["src"]) and np.array_equal(r.dst, ref["dst"])


@pytest.mark.parametrize("bias", ["uniform", "edge_weight", "neighbor_degree"])
@pytest.mark.parametrize("sizes", [[30, 1], [255, 256, 257], [2048, 40], [2049, 40], [1000, 1000]])
def test_rounds_and_table(csaw, bias, sizes):
    g = inputs.rmat_csr(13, 16, 60, 13)
    # one seed, a few, and more frontier vertices than the shared prefix holds
    seeds, io = inputs.distinct_seeds(np.array([1, 7, 64, 3000, 1023, 1024, 1025], dtype=np.uint64), g.V, 4)
    check(csaw, g, seeds, io, sizes, bias)


@pytest.mark.parametrize("cap", [64, 100, 256, 257, None])
@pytest.mark.parametrize("kept", [False, True])
def test_attempts_run_out(csaw, cap, kept):
    # a few edges hold nearly all the weight, so most attempts repeat
    g = inputs.rmat_csr(10, 8, 1, 5)
    w = np.where(np.arange(g.E) % 97 == 0, 1 << 24, 1).astype(np.uint32)
    g = inputs.CSRGraph(g.off, g.col, w)
    seeds, io = inputs.distinct_seeds(np.array([5, 60, 300], dtype=np.uint64), g.V, 6)
    check(csaw, g, seeds, io, [150, 60], "edge_weight", cap, kept)
