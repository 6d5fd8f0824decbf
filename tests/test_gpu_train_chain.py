"""The three chained launches of a training step (zeros, gradient, Adam): the
64-bit and the 128-bit row order, and a captured step against a direct one."""
import pytest
import torch

from paper_1605_02669_gb300 import acs, prior

pytestmark = pytest.mark.gpu

TOTAL, BATCH = 4099, 300


def _trainer(lr=1e-3):
    net = prior.init_params(3)
    g = torch.Generator(device="cuda").manual_seed(7)
    feat = torch.rand((TOTAL, 8), generator=g, device="cuda").bfloat16().view(torch.int16)
    label = (torch.rand(TOTAL, generator=g, device="cuda") < 0.1).float()
    return prior.Trainer(net, lr=lr), feat, label


def _close(x, y, terms):
    # the same addends in another order: at most `terms` FP32 additions, each
    # within 2^-24 of a partial sum that the largest value bounds
    bound = terms * 2.0 ** -24 * max(1.0, float(x.abs().max()))
    return float((x - y).abs().max()) <= bound


@pytest.mark.parametrize("first", [0, 1, TOTAL - BATCH])
@pytest.mark.parametrize("times", [1 << 40, (1 << 62) // TOTAL])
def test_row_order_beyond_64_bits(first, times):
    # a + TOTAL * times walks the same rows as a; its products need 128 bits
    out = []
    for a in (1234, 1234 + TOTAL * times):
        tr, feat, label = _trainer()
        acs.acs_mlp_train_batch(tr.params, feat, label, TOTAL, first, BATCH, a, 17, tr.grad, tr.loss,
                                prior._stream())
        acs.acs_mlp_sync(prior._stream())
        out.append((tr.grad.clone(), tr.loss.clone()))
    assert float(out[0][1]) > 0.0
    assert _close(out[0][0], out[1][0], BATCH) and _close(out[0][1], out[1][1], BATCH)


def test_steps_in_a_graph():
    # a learning rate of zero keeps the weights, so every step's sums compare
    one, feat, label = _trainer(lr=0.0)
    two, _, _ = _trainer(lr=0.0)
    for k in range(3):
        one.batch(feat, label, k * BATCH, BATCH, 1234, 17)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        graph.capture_begin()
        for k in range(3):
            two.batch(feat, label, k * BATCH, BATCH, 1234, 17)
        graph.capture_end()
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(one.params, two.params)
    for x, y in ((one.grad, two.grad), (one.loss, two.loss), (one.m, two.m), (one.v, two.v)):
        assert float(x.abs().max()) > 0.0 and _close(x, y, BATCH)
