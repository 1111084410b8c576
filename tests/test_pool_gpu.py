"""The library's pool keeps the buffers of a large call for the next one, up to
half of the device's memory."""
import numpy as np
import pytest

from paper_2009_09103_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_a_large_calls_buffers_stay():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_09103_gb300 import build
    build.build()
    from paper_2009_09103_gb300 import csaw
    total = torch.cuda.mem_get_info()[1]
    if torch.cuda.mem_get_info()[0] < 0.6 * total:
        pytest.skip("too little device memory free")
    g = inputs.rmat_csr(18, 16, 1, 1)
    G = csaw.Graph(g.off, g.col, None)
    # 4 G edges of eight bytes, and the frontiers and candidates beside them: some 56 GB
    n = 1 << 26
    inst = n >> 13
    seeds = torch.from_numpy(inputs.uniform_vertices(n, g.V, 3).view(np.int32)).cuda()
    io = torch.arange(inst + 1, dtype=torch.int64, device="cuda") * (n // inst)

    def used():
        torch.cuda.synchronize()
        free, all_ = torch.cuda.mem_get_info()
        return all_ - free
    before = used()
    r = csaw.sample(G, seeds, io, [24, 24], "uniform", 1, to_host=False)
    held = used() - before
    del r
    kept = used() - before
    G.close()
    # (memory that is not kept goes back at the waits inside the call already)
    assert held > total // 8 + (2 << 30)
    assert held < total // 2 and kept > 0.98 * held
