"""Order of the stores and reads of one instance's trails across the CTAs of a
cluster, at the sizes where another CTA's store of the same entry is close by.

Every result is bit-identical for every launch shape. The reference is the
oracle, or for restored matrices (which the oracle cannot take) the one-CTA
kernel of acs_iterate_noalloc, which has no second CTA to wait for. A missing
wait loses such a race only now and then: the waits' necessity is derived from
the order of the stores, and these tests run many steps in which it matters.
"""
import numpy as np
import pytest

import oracle
from paper_1605_02669_gb300 import acs, instances

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


# With three to five nodes and tens of ants nearly every closing edge was taken
# by another CTA's ant one step earlier: the closing update has to land on top
# of that ant's store, in both halves of the matrix and in the candidate rows
# (which the next iteration reads).
@pytest.mark.parametrize("n,cl,period", [(3, 2, 1), (3, 1, 1), (4, 3, 1), (5, 2, 1), (4, 2, 2)])
@pytest.mark.parametrize("csize,tpa,m", [(2, 8, 16), (4, 32, 33), (16, 32, 64)])
def test_closing_edge_after_the_step_before(oracle_mod, n, cl, period, csize, tpa, m):
    xy = instances.uniform(n, side=100, seed=n)
    kw = dict(m=m, cl=cl, q0=0.5, seed=12, local_period=period)
    gpu = acs.Colony(xy, acs.params(**kw))
    gpu.set_cluster_size(csize)
    gpu.set_threads_per_ant(tpa)
    ref = oracle.Colony(xy, oracle.make_params(**kw))
    for _ in range(100):
        gpu.run(1)
        ref.run(1)
        for x, y in zip(gpu.tours(), ref.tours()):
            assert np.array_equal(x, y)
        assert np.array_equal(gpu.pheromone().view(np.uint32), ref.pheromone().view(np.uint32))
