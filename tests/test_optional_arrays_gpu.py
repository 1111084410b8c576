"""Search arrays that a caller did not ask for never cost a call its success:
where the caller's allocator has no room beside one, the call gives it back and
goes on without it, with the same result."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu

SCALE = 14


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    g = inputs.rmat_csr(SCALE, 16, 255, 9)
    G = csaw.Graph(g.off, g.col, g.w)
    yield torch, csaw, g, G
    G.use_own_allocator()
    G.close()


class Memory:
    """PyTorch's allocator behind csaw_graph_set_allocator.  An array is a block of
    exactly `array` bytes; while one is held, allocations from the `refuse`-th on
    after it are refused."""

    def __init__(self, env, array):
        self.torch, self.csaw, _, self.G = env
        self.array, self.refuse = array, None
        self.live, self.arrays, self.refused, self.beside = {}, 0, 0, 0
        self.cbs = (self.csaw.ALLOC_FN(self.alloc), self.csaw.FREE_FN(self.free))
        st = self.csaw.lib().csaw_graph_set_allocator(self.G.handle, *self.cbs, None)
        assert st == self.csaw.OK

    def alloc(self, n, stream, ctx):
        if self.array in self.live.values():
            self.beside += 1
            if self.refuse is not None and self.beside >= self.refuse:
                self.refused += 1
                return None
        st = self.torch.cuda.ExternalStream(stream) if stream else None
        p = self.torch.cuda.caching_allocator_alloc(int(n), stream=st)
        self.live[p] = int(n)
        if n == self.array:
            self.arrays, self.beside = self.arrays + 1, 0
        return p

    def free(self, p, stream, ctx):
        del self.live[p]
        self.torch.cuda.caching_allocator_delete(p)

    def check(self, call):
        """call() alike at every place where memory may run out beside the array."""
        ref = call()
        assert self.arrays == 1, "the call is to build an array"
        places = self.beside
        assert places > 0
        for k in range(1, places + 1):
            self.refuse, self.arrays, self.beside, self.refused = k, 0, 0, 0
            got = call()
            assert self.refused > 0 and self.arrays == 1
            assert len(got) == len(ref) and all(np.array_equal(a, b) for a, b in zip(got, ref)), k
            assert not self.live, k
        self.refuse = None


def packed_bytes(g):
    """The packed array: groups and their sums, windows of three 64-edge blocks, a
    record per vertex and a word per chunk of 8192 edges."""
    chunks = -(-g.E // 8192)
    return 8 * (chunks * (8192 + 512 + 1) + 4 * (chunks * 128 // 3 + 1) + 2 * (g.V + 1))


@pytest.mark.parametrize("layer", [False, True])
@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree"])
def test_sampling(env, layer, bias):
    torch, csaw, g, G = env
    mem = Memory(env, packed_bytes(g))
    seeds, io = inputs.distinct_seeds(np.full(300, 20, dtype=np.uint64), g.V, 4)
    call = csaw.layer_sample if layer else csaw.sample

    def run():
        r = call(G, seeds, io, [12, 9], bias, 5)
        return r.edge_offsets, r.frontier_sizes, r.src, r.dst
    mem.check(run)


@pytest.mark.parametrize("instances", [2, 300])
def test_plans(env, instances):
    torch, csaw, g, G = env
    mem = Memory(env, packed_bytes(g))
    seeds, io = inputs.distinct_seeds(np.full(instances, 6000 // instances, dtype=np.uint64), g.V, 4)

    def run():
        plan = csaw.SamplePlan(G, instances, len(seeds), [12, 9], "edge_weight")
        plan.run(seeds, io, 5)
        r = plan.result()
        plan.close()
        return r.edge_offsets, r.frontier_sizes, r.src, r.dst
    mem.check(run)


@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree"])
@pytest.mark.parametrize("build", [False, True])
def test_host_walks(env, bias, build):
    torch, csaw, g, G = env
    mem = Memory(env, packed_bytes(g))
    starts = inputs.uniform_vertices(6000, g.V, 6)

    def run():
        phases = []
        path = csaw.walk(G, starts, 40, bias, 8, build_cdf=build, phase_ms=phases)
        # an array that was asked for is built all the same, by several launches
        # (two events with nothing between are 3 us apart)
        assert not build or phases[0] > 0.008
        return (path,)
    mem.check(run)


def test_node2vec_walks(env):
    torch, csaw, g, G = env
    mem = Memory(env, 8 * (g.E // 2 + g.V + 1))   # the row index: a word of 8 bytes per two edges and per vertex
    starts = inputs.uniform_vertices(3000, g.V, 6)
    mem.check(lambda: (csaw.walk(G, starts, 40, "node2vec", 8, (1, 2, 4)),))


@pytest.mark.parametrize("bias", ["uniform", "edge_weight"])
def test_plan_info_counts_every_buffer(env, bias):
    torch, csaw, g, G = env
    mem = Memory(env, packed_bytes(g))
    plan = csaw.SamplePlan(G, 300, 6000, [12, 9], bias)
    assert mem.arrays == (bias == "edge_weight")
    assert sum(mem.live.values()) == plan.info()["device_bytes"]
    plan.close()
    assert not mem.live


@pytest.mark.parametrize("bias", ["edge_weight", "neighbor_degree"])
@pytest.mark.parametrize("tele", [{}, {"teleport": "restart", "teleport_q32": 1 << 29}])
def test_kept_array_with_zero_biases(env, bias, tele):
    """A kept packed array is searched, not built again, whatever the biases: here zero
    weights, and edges into vertices that have none."""
    torch, csaw, g, _ = env
    off = np.minimum(g.off, g.off[g.V // 2])   # the upper half has no edges of its own
    z = inputs.CSRGraph(off, g.col[:off[-1]], g.w[:off[-1]] & np.uint32(3))
    starts = inputs.uniform_vertices(6000, g.V, 6)
    Z = csaw.Graph(z.off, z.col, z.w)
    mem = Memory((torch, csaw, z, Z), packed_bytes(z))
    Z.build_cdf(bias)
    assert mem.arrays == 1
    got = csaw.walk(Z, starts, 40, bias, 8, **tele)
    assert mem.arrays == 1
    Z.drop_cdf(bias)
    assert np.array_equal(got, csaw.walk(Z, starts, 40, bias, 8, **tele))
    assert mem.arrays == 2
    Z.use_own_allocator()
    Z.close()
    assert np.array_equal(got, oracle.walk(z, starts, 40, bias, 8, **tele))
