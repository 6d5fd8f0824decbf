"""The row order of a training batch on both sides of the line between its
64-bit and its 128-bit remainder."""
import pytest
import torch

from paper_1605_02669_gb300 import acs, prior

pytestmark = pytest.mark.gpu

TOTAL, BATCH, A, C = 4099, 300, 1234, 17


def _gradient(a, first):
    g = torch.Generator(device="cuda").manual_seed(7)
    feat = torch.rand((TOTAL, 8), generator=g, device="cuda").bfloat16().view(torch.int16)
    label = (torch.rand(TOTAL, generator=g, device="cuda") < 0.1).float()
    tr = prior.Trainer(prior.init_params(3))
    acs.acs_mlp_train_batch(tr.params, feat, label, TOTAL, first, BATCH, a, C, tr.grad, tr.loss, prior._stream())
    acs.acs_mlp_sync(prior._stream())
    return tr.grad, tr.loss


# a + TOTAL * times walks the same rows as a. `times`: the largest whose
# products all fit 64 bits, the next, and one far beyond.
@pytest.mark.parametrize("first", [0, 1, TOTAL - BATCH])
@pytest.mark.parametrize("side", ["last below", "first above", "far above"])
def test_rows_are_the_same_on_both_sides(first, side):
    fits = ((1 << 64) - 1 - C) // (first + BATCH)   # the largest a that does
    below = (fits - A) // TOTAL
    times = {"last below": below, "first above": below + 1, "far above": ((1 << 63) - 1 - A) // TOTAL}[side]
    a = A + TOTAL * times
    assert (a * (first + BATCH) + C < 1 << 64) == (side == "last below") and a < 1 << 63
    (g0, l0), (g1, l1) = _gradient(A, first), _gradient(a, first)
    assert float(l0) > 0.0
    # the same addends in another order: at most BATCH FP32 additions, each
    # within 2^-24 of a partial sum that the largest value bounds
    for x, y in ((g0, g1), (l0, l1)):
        assert float((x - y).abs().max()) <= BATCH * 2.0 ** -24 * max(1.0, float(x.abs().max()))
