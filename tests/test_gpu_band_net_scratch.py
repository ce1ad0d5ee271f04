"""The band network under small scratch budgets and with outputs that lie in its
inputs.  Gradients: the shares of the samples that the weight gradients are
summed by shrink to what fits, down to one; another order of a 32-bit sum of
at most 1,024 products is within 1024 * 2^-24 = 6e-5 of its terms' magnitudes
(2^-24 each on average far less): 1e-4 of each block's norm."""
import numpy as np
import pytest

import seqgen

pytestmark = pytest.mark.gpu

H, F = 128, 65
BLOCKS = np.cumsum([0, H * F, H, H * H, H, H, 1])


def _data(n):
    import torch
    rs = seqgen.Stream(400 + n)
    feat = rs.uniform(n * F).reshape(n, F).astype(np.float32)
    target = (3.0 + 4.0 * rs.uniform(n)).astype(np.float32)
    return torch.from_numpy(feat).cuda(), torch.from_numpy(target).cuda()


# activations of n samples take n * 2,056 bytes; 32 shares of sums 3.2 MB more
@pytest.mark.parametrize("n,budget", [(1024, 2105856), (1024, 2500000), (1031, 4200000), (40, 90000)])
def test_gradients_under_a_small_budget(n, budget):
    import torch
    import paper_2412_21103_gb300 as nw
    x, t = _data(n)
    got = []
    for b in (0, budget):
        with nw.Context(0, torch.cuda.current_stream(), mem_budget=b) as ctx:
            nw.nw_band_model_init(ctx, 5)
            grad, loss = nw.nw_band_model_grad(ctx, x, t)
            ctx.sync()
            got.append((grad.cpu().numpy().astype(np.float64), float(loss.item())))
            step = nw.nw_band_model_train_step(ctx, x, t, 1e-3)
            ctx.sync()
            assert abs(float(step.item()) - got[-1][1]) <= 1e-5 * got[-1][1]
    (g, l), (gb, lb) = got
    assert abs(l - lb) <= 1e-5 * l
    for lo, hi in zip(BLOCKS, BLOCKS[1:]):
        assert np.linalg.norm(g[lo:hi] - gb[lo:hi]) <= 1e-4 * np.linalg.norm(g[lo:hi]), (lo, hi)


@pytest.mark.parametrize("at", [0, 20000 * F - 20000, 7 * F])
def test_outputs_that_lie_in_the_inputs(at):
    import torch
    import paper_2412_21103_gb300 as nw
    n = 20000
    x, _ = _data(n)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        nw.nw_band_model_init(ctx, 5)
        want = nw.nw_band_model_forward(ctx, x).clone()
        got = nw.nw_band_model_forward(ctx, x, x.view(-1)[at:at + n])
        ctx.sync()
        assert torch.equal(got, want)
