"""The construct kernel's look-up of a step's edges: lists read whole, four entries
per lane or several times as many, and ants in turns with an index, on both sides
of the lines between them, with many ants on few cities (long chains, edges of
high multiplicity) and on cities whose chains mix. Everything equals the oracle
bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1605_02669_gb300 import acs, instances

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _equal(gpu, ref, memory):
    for x, y in zip(gpu.tours(), ref.tours()):
        assert np.array_equal(x, y)
    a, b = gpu.pheromone(), ref.pheromone()
    for x, y in zip(a, b) if memory else [(a, b)]:
        assert np.array_equal(np.ascontiguousarray(x).view(np.uint32), np.ascontiguousarray(y).view(np.uint32))
    assert gpu.best()[1] == ref.best()[1] and gpu.stats() == ref.stats()


def _run(n, kw, csize, tpa, resident, iters):
    xy = instances.uniform(n, side=40 * n, seed=n)
    gpu = acs.Colony(xy, acs.params(**kw))
    if kw["memory"]:
        gpu.set_spm_resident(resident)
    gpu.set_cluster_size(csize)
    gpu.set_threads_per_ant(tpa)
    ref = oracle.Colony(xy, oracle.make_params(**kw))
    for _ in range(iters):
        gpu.run(1)
        ref.run(1)
        _equal(gpu, ref, kw["memory"])


# m: the last list read whole (four entries per lane), the first looked up, and
# one of several words of the events' order
@pytest.mark.parametrize("memory,resident,period", [(0, 0, 1), (0, 0, 3), (1, 0, 1), (1, 1, 1), (1, 1, 2)])
@pytest.mark.parametrize("csize", [1, 2, 16])
@pytest.mark.parametrize("tpa", [4, 8, 16, 32])
@pytest.mark.parametrize("beyond", [0, 1, 31])
def test_lists_at_the_line(oracle_mod, memory, resident, period, csize, tpa, beyond):
    _run(40, dict(m=4 * tpa + beyond, cl=6, q0=0.8, memory=memory, spm_slots=4, seed=3, local_period=period),
         csize, tpa, resident, 3)


# n = 3: every edge is taken by a third of the ants
@pytest.mark.parametrize("n", [3, 7, 150])
@pytest.mark.parametrize("memory,skip", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("csize,tpa,m", [(1, 4, 256), (1, 16, 1024), (2, 4, 256), (4, 8, 250), (16, 8, 1024),
                                         (16, 32, 1000)])
def test_many_ants_on_few_cities(oracle_mod, n, memory, skip, csize, tpa, m):
    _run(n, dict(m=m, cl=8, q0=0.7, memory=memory, spm_slots=3, seed=5, spm_skip_default=skip), csize, tpa, 1, 2)


# more than four entries per lane, and few enough ants on the cities to read them
@pytest.mark.parametrize("memory,resident,period", [(0, 0, 1), (0, 0, 2), (1, 0, 1), (1, 1, 1), (1, 1, 3)])
@pytest.mark.parametrize("csize,tpa,m,n", [(16, 32, 129, 300), (16, 32, 256, 520), (8, 16, 65, 2600), (4, 16, 66, 300),
                                           (2, 8, 64, 700), (16, 16, 512, 1100)])
def test_long_lists(oracle_mod, memory, resident, period, csize, tpa, m, n):
    _run(n, dict(m=m, cl=10, q0=0.8, memory=memory, spm_slots=4, seed=7, local_period=period), csize, tpa, resident, 2)
