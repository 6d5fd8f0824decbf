"""A relaxed context holds the arrays that its kernels read, and no others."""
import numpy as np
import pytest

from paper_1605_02669_gb300 import acs, instances

pytestmark = pytest.mark.gpu


def test_device_memory_of_a_relaxed_context():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    n, B, m = 500, 1000, 4
    xy = np.concatenate([instances.uniform(n, side=5000, seed=b % 7) for b in range(B)])
    off = np.arange(B + 1, dtype=np.int64) * n
    small = acs.Colony(xy[:n], acs.params(m=m, cl=32, seed=1, relaxed=True))   # loads the module
    small.run(1)
    small.best()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    col = acs.Colony(xy, acs.params(m=m, cl=32, seed=1, relaxed=True), offsets=off)
    used = free0 - torch.cuda.mem_get_info()[0]
    total = n * B
    # per instance n^2 trails and n^2 heuristics; per node coordinates, candidate
    # rows, the tours and the best tour
    needed = 8 * n * n * B + (8 + 256 + 4 * m + 4) * total
    # allocations are rounded up to 2 MB each (fewer than 24 of them); the
    # synchronous kernel's derived data would take 604 bytes a node, 302 MB
    assert used <= needed + 64 * (1 << 20)
    col.run(2)
    tours, lens = col.tours(B - 1)
    assert all(np.array_equal(np.sort(t), np.arange(n)) for t in tours)
    assert col.best(B - 1)[1] <= lens.min()
    col.close()
    small.close()
