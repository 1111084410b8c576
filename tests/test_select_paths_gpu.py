"""Layered selection at the edges of its item classes, bit-exact against the
oracle: whole rows (take_all_kernel up to 1,024 neighbours), short rows (256,
at every alignment), long rows over the packed array, half-warp and whole-warp
fanouts, 32- and 64-bit sums."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu

DEGREES = [1, 2, 5, 15, 16, 17, 31, 33, 63, 100, 248, 249, 255, 256, 257, 300, 1023, 1024, 1025, 3000]


@pytest.fixture(scope="module")
def csaw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw as c
    return c


def graph(wlo, whi, seed=3):
    """8,000 vertices, rows of DEGREES in turn (so rows start at every alignment)."""
    rng = np.random.default_rng(seed)
    V = 8000
    deg = np.array([DEGREES[i % len(DEGREES)] if i < 400 else 1 + i % 6 for i in range(V)])
    cols = [np.sort(rng.choice(V, size=d, replace=False)) for d in deg]
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.uint64)
    return inputs.CSRGraph(off, np.concatenate(cols).astype(np.uint32),
                           rng.integers(wlo, whi + 1, int(off[-1])).astype(np.uint32))


def check(csaw, g, n_inst, fanout, bias, form, cap=None):
    rng = np.random.default_rng(n_inst)
    sizes = rng.integers(1, 120, n_inst)
    seeds = np.concatenate([rng.choice(400, size=s, replace=False) for s in sizes]).astype(np.uint32)
    io = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    kw = {} if cap is None else {"attempt_cap": cap}
    ref = oracle.sample(g, seeds, io, fanout, bias, 9, **kw)
    G = csaw.Graph(g.off, g.col, g.w)
    if form == "kept":
        G.build_cdf(bias)
    r = csaw.sample(G, seeds, io, fanout, bias, 9, attempt_cap=cap)
    plan = csaw.SamplePlan(G, n_inst, len(seeds), fanout, bias, attempt_cap=cap)
    plan.run(seeds, io, 9)
    q = plan.result()
    plan.close()
    G.close()
    for got in (r, q):
        assert np.array_equal(got.edge_offsets, ref["edge_off"])
        assert np.array_equal(got.src, ref["src"]) and np.array_equal(got.dst, ref["dst"])


@pytest.mark.parametrize("bias", ["uniform", "edge_weight", "neighbor_degree"])
@pytest.mark.parametrize("n_inst", [1, 40])
@pytest.mark.parametrize("fanout", [[5, 3], [16, 17], [256, 4], [257, 2], [1024], [1025]])
@pytest.mark.parametrize("form", ["plain", "kept"])
def test_item_classes(csaw, bias, n_inst, fanout, form):
    if form == "kept" and bias == "uniform":
        pytest.skip("uniform bias keeps no array")
    check(csaw, graph(1, 255), n_inst, fanout, bias, form)


# 264 places of 2^24 - 2^18 fit 32 bits, of 2^24 do not; from 2^26 on there is no packed array
@pytest.mark.parametrize("wmax", [2**24 - 2**19, 2**24, 2**26, 2**31])
@pytest.mark.parametrize("form", ["plain", "kept"])
def test_widths(csaw, wmax, form):
    check(csaw, graph(wmax - 1000, wmax), 12, [25, 5], "edge_weight", form)


@pytest.mark.parametrize("cap", [0, 20, 70])
@pytest.mark.parametrize("form", ["plain", "kept"])
def test_updated_sampling(csaw, cap, form):
    check(csaw, graph(1, 3), 12, [25, 5], "edge_weight", form, cap)
