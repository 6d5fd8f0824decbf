"""The construct kernel's waits between CTAs, driven to their limit by a barrier
that never completes: the launch ends, the next read reports ACS_ETIMEOUT, the
context refuses further work, and others are untouched."""
import ctypes
import time

import numpy as np
import pytest

from paper_1605_02669_gb300 import acs, instances

pytestmark = pytest.mark.gpu

HOLD = {"list": 1, "stored": 2, "published": 3}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _batch(sizes, **kw):
    xy = np.concatenate([instances.uniform(n, side=1000, seed=i + 1) for i, n in enumerate(sizes)])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return acs.Colony(xy, acs.params(**kw), offsets=off)


def _runs_out(sizes, m, csize, tpa, memory, period, hold):
    L = acs.load()
    col = _batch(sizes, m=m, cl=6, memory=memory, local_period=period, seed=4)
    col.set_cluster_size(csize)
    col.set_threads_per_ant(tpa)
    col.run(1)
    before = col.best()
    assert L.acs_construct_test_wait_hook(col.ctx, 2 * 10 ** 6, HOLD[hold]) == acs.ACS_OK
    t0 = time.time()
    col.run(2)
    with pytest.raises(acs.AcsError) as e:
        col.best()
    assert e.value.status == acs.ACS_ETIMEOUT and time.time() - t0 < 1.0
    assert L.acs_run_iterations(col.ctx, 1) == acs.ACS_ESTATE
    col.close()
    # a context of the same shape runs as if nothing had been
    again = _batch(sizes, m=m, cl=6, memory=memory, local_period=period, seed=4)
    again.set_cluster_size(csize)
    again.set_threads_per_ant(tpa)
    again.run(1)
    after = again.best()
    assert before[1] == after[1] and np.array_equal(before[0], after[0])
    again.close()


# the last: more instances than clusters are resident, so clusters would draw more
@pytest.mark.parametrize("sizes,m,csize,tpa", [([90], 20, 2, 8), ([90], 33, 4, 32), ([90, 40], 64, 16, 16),
                                               ([70, 50, 30] * 130, 8, 2, 32)])
@pytest.mark.parametrize("memory,period", [(0, 1), (0, 3), (1, 1)])
@pytest.mark.parametrize("hold", sorted(HOLD))
def test_a_wait_that_runs_out_ends_the_launch(sizes, m, csize, tpa, memory, period, hold):
    _runs_out(sizes, m, csize, tpa, memory, period, hold)


# the variants for more than four list entries per lane, on both ways of voting
@pytest.mark.parametrize("n,m,csize,tpa,memory", [(700, 64, 2, 8, 0), (600, 256, 16, 32, 0), (600, 256, 16, 32, 1)])
@pytest.mark.parametrize("hold", sorted(HOLD))
def test_a_wait_that_runs_out_on_long_lists(n, m, csize, tpa, memory, hold):
    _runs_out([n], m, csize, tpa, memory, 1, hold)


@pytest.mark.parametrize("memory", [0, 1])
@pytest.mark.parametrize("csize,tpa,m", [(1, 16, 40), (4, 8, 256)])
def test_kernels_with_barriers_do_not_wait(memory, csize, tpa, m):
    L = acs.load()
    col = _batch([60], m=m, cl=6, memory=memory, seed=4)
    col.set_cluster_size(csize)
    col.set_threads_per_ant(tpa)
    assert L.acs_construct_test_wait_hook(col.ctx, 10 ** 6, HOLD["list"]) == acs.ACS_OK
    col.run(2)
    assert col.best()[1] > 0
    col.close()


def test_the_hook_can_be_taken_back_and_checks_its_arguments():
    L = acs.load()
    col = _batch([80], m=32, cl=6, seed=4)
    col.set_cluster_size(4)
    for ns, hold in ((-1, 0), (0, -1), (0, 4)):
        assert L.acs_construct_test_wait_hook(col.ctx, ns, hold) == acs.ACS_EINVAL
    assert L.acs_construct_test_wait_hook(ctypes.c_void_p(), 0, 0) == acs.ACS_EINVAL
    assert L.acs_construct_test_wait_hook(col.ctx, 10 ** 6, HOLD["list"]) == acs.ACS_OK
    assert L.acs_construct_test_wait_hook(col.ctx, 0, 0) == acs.ACS_OK
    col.run(3)
    assert col.best()[1] > 0
    col.close()
