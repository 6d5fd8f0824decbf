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


# With three to five nodes nearly every closing edge was taken by another CTA's ant
# one step earlier (up to a dozen ants do not take turns on 8 and 16 CTAs): the closing update has to land on top
# of that ant's store, in both halves of the matrix and in the candidate rows
# (which the next iteration reads).
@pytest.mark.parametrize("n,cl,period", [(3, 2, 1), (3, 1, 1), (4, 3, 1), (5, 2, 1), (4, 2, 2)])
@pytest.mark.parametrize("csize,tpa,m", [(2, 8, 16), (4, 32, 33), (16, 32, 64), (16, 32, 9), (16, 8, 12), (8, 4, 7)])
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


def _restored(n, m, cl, period, rng, kind):
    """A context's image after two iterations with some trails of the matrix
    replaced, and the same state in the caller's buffers of acs_iterate_noalloc."""
    import torch

    xy = instances.uniform(n, side=60, seed=n)
    p = acs.params(m=m, cl=cl, q0=0.7, seed=6, local_period=period)
    col = acs.Colony(xy, p)
    col.run(2)
    nn, w, tau0, _ = col.setup()
    tau = col.pheromone().copy()
    if kind == "overflow":   # more than 32 changed trails in every row
        i, j = np.repeat(np.arange(n), 48), rng.integers(0, n, 48 * n)
        f = rng.uniform(1.0, 4.0, i.size)
    else:                    # a few below tau0 in every row
        i, j = np.repeat(np.arange(n), 3), rng.integers(0, n, 3 * n)
        f = rng.uniform(0.3, 1.0, i.size)
    tau[i, j] = (float(tau0) * f).astype(np.float32)
    tau = np.minimum(tau, tau.T) if kind == "low" else np.maximum(tau, tau.T)
    buf = col.get_state()
    at = 128 + 256 * n + 4 * n
    buf[at:at + 4 * n * n] = tau.reshape(-1).view(np.uint8)
    best, best_len = col.best()
    nn32, w32 = np.full((n, 32), -1, np.int32), np.zeros((n, 32), np.float32)
    nn32[:, :nn.shape[1]], w32[:, :nn.shape[1]] = nn, w
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in dict(
        xy=xy, nn=nn32, w=w32, tau=tau, best=best.astype(np.int32), best_len=np.array([best_len], np.int64),
        tours=np.zeros((m, n), np.int32), lens=np.zeros(m, np.int64)).items()}
    torch.cuda.synchronize()
    return xy, p, buf, float(tau0), nn.shape[1], dev


# One candidate: an ant reads its whole row in nearly every step, and the row's
# trails were stored by other CTAs one and two lists earlier.
@pytest.mark.parametrize("kind", ["overflow", "low"])
@pytest.mark.parametrize("csize,tpa,m,period", [(2, 8, 24, 1), (4, 32, 40, 1), (16, 32, 96, 1), (8, 16, 64, 3)])
def test_whole_rows_are_read_behind_their_updates(kind, csize, tpa, m, period):
    import torch

    n = 150
    xy, p, buf, tau0, cl, d = _restored(n, m, 1, period, np.random.default_rng(9), kind)
    gpu = acs.Colony(xy, p)
    gpu.set_cluster_size(csize)
    gpu.set_threads_per_ant(tpa)
    gpu.set_state(buf)
    for it in range(2, 22):
        rc = acs.acs_iterate_noalloc(d["xy"].data_ptr(), n, d["nn"].data_ptr(), d["w"].data_ptr(), cl, tau0,
                                     d["tau"].data_ptr(), d["tours"].data_ptr(), d["lens"].data_ptr(),
                                     d["best"].data_ptr(), d["best_len"].data_ptr(), it, p,
                                     torch.cuda.current_stream().cuda_stream)
        assert rc == acs.ACS_OK
        gpu.run(1)
        t, L = gpu.tours()
        assert np.array_equal(d["tours"].cpu().numpy(), t) and np.array_equal(d["lens"].cpu().numpy(), L)
        assert gpu.best()[1] == int(d["best_len"].cpu()[0])
        assert np.array_equal(d["tau"].cpu().numpy().view(np.uint32), gpu.pheromone().view(np.uint32))


# Trails and records that another CTA's publication makes visible, on the
# matrix, in global memory and in distributed shared memory: many ants on few
# nodes, so that nearly every read is of something just stored elsewhere.
@pytest.mark.parametrize("memory,resident", [(0, None), (1, 0), (1, 1)])
@pytest.mark.parametrize("csize,tpa", [(2, 4), (4, 16), (16, 32)])
def test_published_updates_are_seen_by_other_ctas(memory, resident, csize, tpa):
    xy = instances.uniform(48, side=200, seed=5)
    kw = dict(m=64, cl=10, q0=0.8, memory=memory, spm_slots=4, seed=31)
    cols = [acs.Colony(xy, acs.params(**kw)) for _ in range(2)]
    for col, (c, t) in zip(cols, ((1, 8), (csize, tpa))):
        if resident is not None:
            col.set_spm_resident(resident)
        col.set_cluster_size(c)
        col.set_threads_per_ant(t)
    for _ in range(10):
        for col in cols:
            col.run(20)
        for x, y in zip(cols[0].tours(), cols[1].tours()):
            assert np.array_equal(x, y)
        a, b = (col.pheromone() for col in cols)
        for x, y in zip(a, b) if memory else [(a, b)]:
            assert np.array_equal(np.ascontiguousarray(x).view(np.uint32), np.ascontiguousarray(y).view(np.uint32))
        assert cols[0].stats() == cols[1].stats()
