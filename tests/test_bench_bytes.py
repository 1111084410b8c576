"""The byte model of walks over the packed array, against a count step by step."""
import numpy as np
import pytest


def test_packed_walk_bytes():
    torch = pytest.importorskip("torch")
    import bench
    NONE = 0xFFFFFFFF
    path = np.array([[0, 1, 2, 0], [3, NONE, NONE, NONE], [2, 1, NONE, NONE]], dtype=np.uint32)
    L = path.shape[1] - 1
    want = 0
    for row in path:
        want += 4 + 4 * (L + 1)   # start, path row
        for b in row[1:]:
            if b == NONE:
                break
            # two records, a window of block ends, a block's group sums, the group's biases and columns, the entry
            want += 32 + 32 + 32 + 64 + 4
    got = bench.packed_walk_bytes(torch, torch.tensor([0, 1, 3, 4, 4]), torch.from_numpy(path.view(np.int32)), L)
    assert got == want
