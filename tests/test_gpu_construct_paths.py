"""The construct kernel's rarer paths on the GPU, at the sizes where they begin.

Ants in turns (more ants in a CTA than groups of lanes), the search for the
nearest unvisited node beyond a city's list of boxes and with equal keys, and,
on restored matrices, rows whose changed trails are listed, do not fit the
list, lie below tau0 or differ between the two halves. Every result is
bit-identical for every launch shape; the reference is the oracle, or for
restored matrices (which the oracle cannot take) the one-CTA kernel of
acs_iterate_noalloc, which reads every trail from the matrix.
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


def _same(gpu, ref, memory):
    tg, lg = gpu.tours()
    tr, lr = ref.tours()
    assert np.array_equal(tg, tr) and np.array_equal(lg, lr)
    assert gpu.best()[1] == ref.best()[1]
    if memory == 0:
        assert np.array_equal(gpu.pheromone().view(np.uint32), ref.pheromone().view(np.uint32))
    else:
        gv, gi, gt = gpu.pheromone()
        rv, ri, rt = ref.pheromone()
        assert np.array_equal(gi, ri) and np.array_equal(gt, rt)
        assert np.array_equal(gv.view(np.uint32), rv.view(np.uint32))
    assert gpu.stats() == ref.stats()


# ants per CTA x lanes above 1024 (one CTA) or 512 (clusters): turns; just below: not
@pytest.mark.parametrize("csize,tpa,m", [(1, 32, 32), (1, 32, 33), (1, 8, 300), (2, 32, 33), (4, 16, 128),
                                         (4, 16, 131), (8, 32, 270), (2, 8, 129)])
@pytest.mark.parametrize("memory,period", [(0, 1), (0, 3), (1, 1), (1, 2)])
def test_ants_in_turns_and_at_the_edge(oracle_mod, csize, tpa, m, memory, period):
    xy = instances.clustered(150, seed=41)
    kw = dict(m=m, cl=8, q0=0.8, memory=memory, spm_slots=5, seed=3, local_period=period)
    gpu = acs.Colony(xy, acs.params(**kw))
    gpu.set_cluster_size(csize)
    gpu.set_threads_per_ant(tpa)
    ref = oracle.Colony(xy, oracle.make_params(**kw))
    for _ in range(2):
        gpu.run(1)
        ref.run(1)
        _same(gpu, ref, memory)


# 32 boxes of 32 nodes are listed per city: n = 1024 is the last size whose list
# holds all boxes. One candidate makes empty candidate sets the rule; beta 0 and
# 8 and duplicated points make equal keys.
@pytest.mark.parametrize("n,beta", [(1024, 2), (1025, 2), (1300, 2), (1300, 0), (1300, 8)])
@pytest.mark.parametrize("csize,tpa,memory", [(1, 8, 0), (2, 32, 0), (1, 16, 1), (4, 4, 1)])
def test_nearest_node_search(oracle_mod, n, beta, csize, tpa, memory):
    base = instances.uniform(n - 100, side=900, seed=n)
    xy = np.concatenate([base, base[:100]]).astype(np.int32)
    kw = dict(m=9, cl=1, q0=0.9, beta=beta, memory=memory, spm_slots=3, seed=8)
    gpu = acs.Colony(xy, acs.params(**kw))
    gpu.set_cluster_size(csize)
    gpu.set_threads_per_ant(tpa)
    ref = oracle.Colony(xy, oracle.make_params(**kw))
    for _ in range(2):
        gpu.run(1)
        ref.run(1)
        _same(gpu, ref, memory)


def _doctored(kind, tau, tau0, rng):
    n = tau.shape[0]
    t = tau.copy()
    if kind == "listed":        # a few raised trails, both halves
        i, j = rng.integers(0, n, 3 * n), rng.integers(0, n, 3 * n)
    elif kind == "overflow":    # more than 32 in some rows
        i, j = np.repeat(np.arange(6), 60), rng.integers(0, n, 360)
    else:
        i, j = rng.integers(0, n, n), rng.integers(0, n, n)
    f = rng.uniform(0.2, 30.0, i.size) if kind == "low" else rng.uniform(1.0, 30.0, i.size)
    v = (tau0 * f).astype(np.float32)
    t[i, j] = v
    if kind != "halves":
        t[j, i] = v
    return t


@pytest.mark.parametrize("kind", ["listed", "overflow", "low", "halves"])
@pytest.mark.parametrize("csize,tpa,m", [(1, 8, 24), (4, 32, 24), (2, 4, 25), (1, 32, 40), (8, 16, 70)])
def test_restored_matrix_equals_the_plain_kernel(kind, csize, tpa, m):
    import torch

    n = 120
    xy = instances.uniform(n, side=1000, seed=51)
    p = acs.params(m=m, cl=4, q0=0.7, seed=6)
    col = acs.Colony(xy, p)
    col.run(2)
    nn, w, tau0, _ = col.setup()
    tau = _doctored(kind, col.pheromone(), float(tau0), np.random.default_rng(7))
    buf = col.get_state()
    at = 128 + 256 * n + 4 * n
    buf[at:at + 4 * n * n] = tau.reshape(-1).view(np.uint8)
    best, best_len = col.best()
    dev = torch.device("cuda:0")
    cl = nn.shape[1]
    nn32 = np.full((n, 32), -1, np.int32)
    w32 = np.zeros((n, 32), np.float32)
    nn32[:, :cl], w32[:, :cl] = nn, w
    d = {k: torch.from_numpy(np.ascontiguousarray(v)).to(dev)
         for k, v in dict(xy=xy, nn=nn32, w=w32, tau=tau, best=best.astype(np.int32),
                          best_len=np.array([best_len], np.int64)).items()}
    d["tours"] = torch.zeros((m, n), dtype=torch.int32, device=dev)
    d["lens"] = torch.zeros(m, dtype=torch.int64, device=dev)
    torch.cuda.synchronize()
    gpu = acs.Colony(xy, p)
    gpu.set_cluster_size(csize)
    gpu.set_threads_per_ant(tpa)
    gpu.set_state(buf)
    for it in (2, 3):
        rc = acs.acs_iterate_noalloc(d["xy"].data_ptr(), n, d["nn"].data_ptr(), d["w"].data_ptr(), cl, float(tau0),
                                     d["tau"].data_ptr(), d["tours"].data_ptr(), d["lens"].data_ptr(),
                                     d["best"].data_ptr(), d["best_len"].data_ptr(), it, p,
                                     torch.cuda.current_stream(dev).cuda_stream)
        assert rc == acs.ACS_OK
        gpu.run(1)
        t, L = gpu.tours()
        assert np.array_equal(d["tours"].cpu().numpy(), t) and np.array_equal(d["lens"].cpu().numpy(), L)
        assert gpu.best()[1] == int(d["best_len"].cpu()[0])
        assert np.array_equal(d["tau"].cpu().numpy().view(np.uint32), gpu.pheromone().view(np.uint32))


# Batches that share the SMs: whatever shape the context starts with, every best
# tour is that of clusters of four CTAs, and the first and last instance's tours
# are the oracle's.
@pytest.mark.parametrize("memory", [0, 1])
@pytest.mark.parametrize("m,sizes", [
    (8, [40] * 90), (20, [33, 64, 65, 300] * 25), (32, [700] * 8 + [60] * 100), (48, [100] * 160),
    (64, [50] * 310), (64, [1500] * 2 + [70] * 90), (65, [48] * 80), (130, [40] * 80)])
def test_default_shape_of_a_batch(oracle_mod, memory, m, sizes):
    parts = [instances.uniform(n, seed=i + 1) for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    kw = dict(m=m, memory=memory, seed=11)
    a = acs.Colony(np.concatenate(parts), acs.params(**kw), offsets=off)
    b = acs.Colony(np.concatenate(parts), acs.params(**kw), offsets=off)
    assert (a.cluster_size, a.threads_per_ant) in {(1, 8), (1, 16), (1, 32), (2, 8), (2, 16)}
    b.set_cluster_size(4)
    b.set_threads_per_ant(8)
    for col in (a, b):
        col.run(2)
    for i in range(len(sizes)):
        ta, la = a.best(i)
        tb, lb = b.best(i)
        assert la == lb and np.array_equal(ta, tb)
    for i in (0, len(sizes) - 1):
        ref = oracle.Colony(parts[i], oracle.make_params(**kw), instance=i)
        ref.run(2)
        for x, y in zip(a.tours(i), ref.tours()):
            assert np.array_equal(x, y)
    a.close()
    b.close()
