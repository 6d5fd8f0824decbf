"""acs_iterate_noalloc on coordinates outside [0, 2^20): its buffers are the
caller's, and nothing limits them to the range that acs_create checks."""
import math

import numpy as np
import pytest

from paper_1605_02669_gb300 import acs

pytestmark = pytest.mark.gpu


def _distances(xy):
    """nint of the exact Euclidean distances, by integer square roots."""
    n = len(xy)
    d = np.zeros((n, n), np.int64)
    for i in range(n):
        for j in range(n):
            s = int(xy[i, 0] - xy[j, 0]) ** 2 + int(xy[i, 1] - xy[j, 1]) ** 2
            r = math.isqrt(s)
            d[i, j] = r + (1 if s - r * r > r else 0)
    return d


# lo, hi: a range of the same width below zero, one just past 2^20, and wide ones
@pytest.mark.parametrize("lo,hi", [(-500000, 500000), (0, 1 << 20), (-(1 << 20), 1 << 20), (-3000000, 5000000),
                                   (-500000000, 500000000)])
def test_tours_and_lengths(lo, hi):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    n, m = 60, 8
    rng = np.random.default_rng(abs(lo) + hi)
    xy = rng.integers(lo, hi, (n, 2), dtype=np.int64)
    xy[0], xy[1] = (lo, lo), (hi, hi)
    d = _distances(xy)
    far = np.where(np.eye(n, dtype=bool), np.int64(1) << 40, d)
    nn = np.lexsort((np.arange(n)[None, :].repeat(n, 0), far))[:, :1]
    # one candidate and q0 = 1: on a matrix of tau0 every choice is the largest
    # weight, 1 / d^2 in FP32, ties to the lowest node
    x = np.maximum(d, 1).astype(np.float32)
    w = np.float32(1) / (x * x)
    tau0 = np.float32(0.25)
    p = acs.params(m=m, cl=1, q0=1.0, beta=2, seed=2)
    nn32, w32 = np.full((n, 32), -1, np.int32), np.zeros((n, 32), np.float32)
    nn32[:, :1], w32[:, :1] = nn, np.take_along_axis(w, nn, 1)
    b = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in dict(
        xy=xy.astype(np.int32), nn=nn32, w=w32, tau=np.full((n, n), tau0), tours=np.zeros((m, n), np.int32),
        lens=np.zeros(m, np.int64), best=np.zeros(n, np.int32),
        best_len=np.array([np.iinfo(np.int64).max])).items()}
    torch.cuda.synchronize()
    rc = acs.acs_iterate_noalloc(b["xy"].data_ptr(), n, b["nn"].data_ptr(), b["w"].data_ptr(), 1, float(tau0),
                                 b["tau"].data_ptr(), b["tours"].data_ptr(), b["lens"].data_ptr(),
                                 b["best"].data_ptr(), b["best_len"].data_ptr(), 0, p,
                                 torch.cuda.current_stream().cuda_stream)
    assert rc == acs.ACS_OK
    tours, lens = b["tours"].cpu().numpy(), b["lens"].cpu().numpy()
    for a in range(m):
        left, c, tour = set(range(n)), int(tours[a, 0]), []
        for _ in range(n):
            tour.append(c)
            left.discard(c)
            if not left:
                break
            k = int(nn[c, 0])
            # the full scan's products carry the trail: tau0 * weight, rounded
            c = k if k in left else max(left, key=lambda j: (tau0 * w[c, j], -j))
        assert np.array_equal(tours[a], tour)
        assert int(lens[a]) == sum(int(d[tour[i], tour[(i + 1) % n]]) for i in range(n))
    assert int(b["best_len"].cpu()[0]) == int(lens.min())
