"""Frontiers built by one block and by the device-wide kernels, bit-exact
against the oracle on both sides of the sizes where the paths change: seeds and
picks around 4,096, frontier positions around 8,192, sorts around 131,072 keys,
empty instances, duplicate seeds and errors."""
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


@pytest.mark.parametrize("n_seeds", [1, 31, 33, 1023, 4095, 4096, 4097, 8192, 8193, 131000, 131200])
@pytest.mark.parametrize("n_inst", [1, 3, 5000])
def test_sizes(csaw, n_seeds, n_inst):
    g = inputs.rmat_csr(11, 6, 20, 2)
    rng = np.random.default_rng(n_seeds)
    seeds = rng.integers(0, g.V, n_seeds).astype(np.uint32)   # duplicates among them
    # instances of unequal size, empty ones among them
    io = np.concatenate([[0], np.sort(rng.integers(0, n_seeds + 1, n_inst - 1)), [n_seeds]]).astype(np.uint64)
    fanout = [1, 2, 1]
    ref = oracle.sample(g, seeds, io, fanout, "edge_weight", 5)
    G = csaw.Graph(g.off, g.col, g.w)
    r = csaw.sample(G, seeds, io, fanout, "edge_weight", 5)
    plan = csaw.SamplePlan(G, n_inst, n_seeds, fanout, "edge_weight")
    plan.run(seeds, io, 5)
    q = plan.result()
    plan.close()
    G.close()
    for got in (r, q):
        assert np.array_equal(got.edge_offsets, ref["edge_off"])
        assert np.array_equal(got.frontier_sizes, ref["fsize"][:len(got.frontier_sizes)])
        assert np.array_equal(got.src, ref["src"]) and np.array_equal(got.dst, ref["dst"])


@pytest.mark.parametrize("n_seeds", [100, 5000])
def test_device_input_errors(csaw, n_seeds):
    import torch
    g = inputs.rmat_csr(8, 8, 20, 2)
    G = csaw.Graph(g.off, g.col, g.w)

    def dev(a, t):
        return torch.from_numpy(a.astype(t)).cuda()
    good = np.zeros(n_seeds)
    bad = good.copy()
    bad[n_seeds // 2] = g.V
    for seeds, io in ((bad, [0, n_seeds]), (good, [1, n_seeds]), (good, [0, n_seeds, n_seeds - 1, n_seeds])):
        with pytest.raises(csaw.CsawError) as e:
            csaw.sample(G, dev(seeds, np.int32), dev(np.array(io), np.int64), [2], "uniform", 1)
        assert e.value.status == csaw.ERR_INVALID
    G.close()
