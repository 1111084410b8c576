"""Served sampling requests batched together whose fanouts differ: whole rows
(FANOUT_ALL) beside draws of more picks than a warp's list holds, each result
that of the oracle for the request alone."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu


# bias, weights (smallest, largest), cumulative array kept; hub: its degree, within a
# block's shared memory and past it.  Zero weights draw from shared hub arrays, positive ones
# from the packed array, weights of 2^26 and more from the cumulative array alone
@pytest.mark.parametrize("bias,wlo,whi,kept", [
    ("uniform", 1, 9, False), ("edge_weight", 1, 255, False), ("edge_weight", 0, 3, False),
    ("edge_weight", 1, 255, True), ("edge_weight", 1, 1 << 27, True), ("neighbor_degree", 1, 1, False)])
@pytest.mark.parametrize("hub", [5000, 9001])
def test_whole_rows_beside_many_picks(bias, wlo, whi, kept, hub):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    rng = np.random.default_rng(hub)
    V = 10000
    pairs = np.concatenate([np.stack([np.full(n, h), 4 + rng.choice(V - 4, size=n, replace=False)], 1)
                            for h, n in enumerate((hub, 700, 301, 90))])
    a = np.unique(np.concatenate([pairs, pairs[:, ::-1]]), axis=0)
    off = np.zeros(V + 1, dtype=np.uint64)
    off[1:] = np.cumsum(np.bincount(a[:, 0], minlength=V))
    g = inputs.CSRGraph(off, a[:, 1].astype(np.uint32), rng.integers(wlo, whi + 1, size=len(a)).astype(np.uint32))
    G = csaw.Graph(g.off, g.col, g.w)
    if kept:
        G.build_cdf(bias)
    fans = [[csaw.FANOUT_ALL], [300], [csaw.FANOUT_ALL, 2], [300, 300], [7, csaw.FANOUT_ALL], [257, 1, 2]]
    seeds = np.array([0, 1, 2, 3, 17, 0, 3], dtype=np.uint32)
    io = np.array([0, 5, 5, 7], dtype=np.uint64)
    srv = csaw.Server(G, budget_bytes=8 << 30, slots=1)
    busy = srv.submit_walk(inputs.uniform_vertices(1 << 18, V, 7), 400, "uniform", 1)   # the slot's work meanwhile
    tickets = [srv.submit_sample(seeds, io, f, bias, 50 + i) for i, f in enumerate(fans)]
    srv.poll(busy)
    got = [srv.poll(t) for t in tickets]
    srv.close()
    G.close()
    assert len({r.t_admit_ns for r in got}) == 1   # one batch
    for i, (f, r) in enumerate(zip(fans, got)):
        ref = oracle.sample(g, seeds, io, f, bias, 50 + i)
        assert np.array_equal(r.sample.edge_offsets, ref["edge_off"]), f
        assert np.array_equal(r.sample.src, ref["src"]) and np.array_equal(r.sample.dst, ref["dst"]), f
