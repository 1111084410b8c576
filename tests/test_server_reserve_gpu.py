"""The admission budget is charged for an array only where the batch builds one:
requests that fit the budget side by side run side by side otherwise."""
import numpy as np
import pytest

import oracle
from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["walk", "sample"])
@pytest.mark.parametrize("case", ["kept", "unweighted", "wide", "zero"])
def test_nothing_reserved_for_no_array(case, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if (case, kind) == ("zero", "walk"):
        pytest.skip("walks over zero weights build the array")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    g = inputs.rmat_csr(15, 16, 255, 21)
    w = {"kept": g.w, "unweighted": None, "wide": g.w << np.uint32(20), "zero": g.w & np.uint32(3)}[case]
    g = inputs.CSRGraph(g.off, g.col, w)
    G = csaw.Graph(g.off, g.col, g.w)
    if case == "kept":
        G.build_cdf("edge_weight")
    array = 9 * g.E
    starts = inputs.uniform_vertices(60000, g.V, 2)
    seeds, io = inputs.distinct_seeds(np.full(40, 300, dtype=np.uint64), g.V, 4)

    def submit(srv, k):
        if kind == "walk":
            return srv.submit_walk(starts, 80, "edge_weight", k)
        return srv.submit_sample(seeds, io, [10, 10], "edge_weight", k)
    srv = csaw.Server(G, budget_bytes=8 << 30, slots=1)
    one = srv.poll(submit(srv, 0)).estimate
    srv.close()
    # two requests fit, two and an array do not; an array fits a slot's share
    budget = 2 * one + array // 2
    assert budget // 4 > array
    srv = csaw.Server(G, budget_bytes=budget, slots=2, max_batch=1)
    got = [srv.poll(t) for t in [submit(srv, k) for k in range(12)]]
    srv.close()
    G.close()
    spans = sorted((r.t_admit_ns, r.t_finish_ns) for r in got)
    assert any(b[0] < a[1] for a, b in zip(spans, spans[1:]))
    for k in (0, 11):
        if kind == "walk":
            assert np.array_equal(got[k].path, oracle.walk(g, starts, 80, "edge_weight", k))
        else:
            ref = oracle.sample(g, seeds, io, [10, 10], "edge_weight", k)
            assert np.array_equal(got[k].sample.src, ref["src"]) and np.array_equal(got[k].sample.dst, ref["dst"])
