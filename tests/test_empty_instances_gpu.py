"""Few seeds among very many instances, most of them empty: what goes through
the instances is spread over the chip, and the results stay the oracle's."""
import time

import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    return torch, csaw


# either side of the largest count that one block goes through, and well past it
@pytest.mark.parametrize("n_inst", [4095, 4096, 4097, 70001])
@pytest.mark.parametrize("n_seeds", [1, 700, 4097])
@pytest.mark.parametrize("layer", [False, True])
def test_results(env, n_inst, n_seeds, layer):
    torch, csaw = env
    g = inputs.rmat_csr(10, 8, 20, 2)
    rng = np.random.default_rng(n_inst + n_seeds)
    seeds = rng.integers(0, g.V, n_seeds).astype(np.uint32)
    io = np.concatenate([[0], np.sort(rng.integers(0, n_seeds + 1, n_inst - 1)), [n_seeds]]).astype(np.uint64)
    ref = oracle.sample(g, seeds, io, [2, 3], "edge_weight", 5, layer=layer)
    G = csaw.Graph(g.off, g.col, g.w)
    got = [(csaw.layer_sample if layer else csaw.sample)(G, seeds, io, [2, 3], "edge_weight", 5)]
    if not layer:
        plan = csaw.SamplePlan(G, n_inst, n_seeds, [2, 3], "edge_weight")
        plan.run(seeds, io, 5)
        got.append(plan.result())
        plan.close()
    G.close()
    for r in got:
        assert np.array_equal(r.edge_offsets, ref["edge_off"])
        assert np.array_equal(r.frontier_sizes, ref["fsize"][:len(r.frontier_sizes)])
        assert np.array_equal(r.src, ref["src"]) and np.array_equal(r.dst, ref["dst"])


def test_time(env):
    """Two million instances are 32 MB of offsets and sizes a layer, some 10 us at memory's
    rate; one block alone takes over 1 ms to go through them once."""
    torch, csaw = env
    g = inputs.rmat_csr(12, 8, 20, 2)
    G = csaw.Graph(g.off, g.col, g.w)
    n = 2000000
    io = torch.full((n + 1,), 100, dtype=torch.int64, device="cuda")
    io[0] = 0
    seeds = torch.from_numpy(inputs.uniform_vertices(100, g.V, 3).view(np.int32)).cuda()
    plan = csaw.SamplePlan(G, n, 100, [5, 5], "edge_weight")
    times = []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        plan.run(seeds, io, 1)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    plan.close()
    G.close()
    assert min(times) < 1.0, times


def test_reading_the_offsets(env):
    """The offsets and sizes of two million instances are read about as fast as their bytes
    are copied into the same kind of host memory."""
    torch, csaw = env
    g = inputs.rmat_csr(12, 8, 20, 2)
    G = csaw.Graph(g.off, g.col, g.w)
    n = 2000000
    seeds, io = inputs.uniform_vertices(100, g.V, 3), np.full(n + 1, 100, dtype=np.uint64)
    io[0] = 0
    plan = csaw.SamplePlan(G, n, 100, [5, 5], "edge_weight")
    words = torch.zeros(4 * n, dtype=torch.int64, device="cuda")
    host = torch.zeros(4 * n, dtype=torch.int64)
    read, copy = [], []
    for _ in range(6):
        plan.run(seeds, io, 1)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        plan.n_edges()
        t1 = time.perf_counter()
        host.copy_(words)
        read.append(t1 - t0)
        copy.append(time.perf_counter() - t1)
    plan.close()
    G.close()
    assert min(read) < 1.6 * min(copy), (read, copy)
