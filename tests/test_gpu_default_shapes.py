"""What a context starts with when many ants or many instances share the GPU, and
that a batch's tours do not depend on it."""
import numpy as np
import pytest

from paper_1605_02669_gb300 import acs, instances

pytestmark = pytest.mark.gpu


def _colony(B, n, m, memory):
    xy = np.concatenate([instances.uniform(n, side=20 * n, seed=b + 1) for b in range(B)])
    return acs.Colony(xy, acs.params(m=m, cl=16, memory=memory, seed=2), offsets=np.arange(B + 1, dtype=np.int64) * n)


# clusters of two and more never start with four lanes per ant; an SPM's records
# are in shared memory where all instances run at once all the same
@pytest.mark.parametrize("memory", [0, 1])
@pytest.mark.parametrize("B,n,m", [(1, 50, 1024), (1, 300, 256), (16, 400, 128), (60, 200, 256), (100, 150, 40),
                                   (200, 200, 64), (200, 100, 200)])
def test_defaults(memory, B, n, m):
    import __graft_entry__

    __graft_entry__.build()
    a, b = _colony(B, n, m, memory), _colony(B, n, m, memory)
    assert a.threads_per_ant >= 8
    if memory:
        assert a.kernel_mode == 2
        b.set_spm_resident(0)
    b.set_cluster_size(2)
    b.set_threads_per_ant(16)
    for col in (a, b):
        col.run(2)
    for i in (0, B // 2, B - 1):
        for x, y in zip(a.tours(i), b.tours(i)):
            assert np.array_equal(x, y)
        assert a.best(i)[1] == b.best(i)[1] and a.stats(i) == b.stats(i)
    a.close()
    b.close()
