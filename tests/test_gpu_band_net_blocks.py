"""Gradients of the band network block by block (each layer's weights and biases
come from blocks and shares of their own), against the float64 reference with
the same BF16 roundings.  Tolerance: 32-bit sums of at most 128 products are
within 128 * 2^-24 = 8e-6 of their terms, which moves an activation to the
other side of a BF16 rounding (2^-8 of itself) with a chance of about 8e-6 * 2^8 =
2e-3, so a block's relative error is about sqrt(2e-3) * 2^-8 = 2e-4 per
layer it passes; 2e-3 of each block's norm.  A unit group or a share left out is
at least 1 / 33 of the samples or 1 / 8 of a block: 3e-2 and more.  The loss is
a mean of squares of outputs with errors far below 1e-3 of them."""
import numpy as np
import pytest

import seqgen
from oracle import band_model as bm

pytestmark = pytest.mark.gpu

H, F = 128, 65
SIZES = [("W1", H * F), ("b1", H), ("W2", H * H), ("b2", H), ("W3", H), ("b3", 1)]


# one share; two; 33 samples a share and a last one of 8; 47 and a last one of 43
@pytest.mark.parametrize("n", [32, 33, 1031, 1500])
def test_each_block_of_the_gradients(n):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(900 + n)
    feat = rs.uniform(n * F).reshape(n, F).astype(np.float32)
    target = (3.0 + 4.0 * rs.uniform(n)).astype(np.float32)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        nw.nw_band_model_init(ctx, 6)
        params = nw.nw_band_model_get(ctx)
        grad, loss = nw.nw_band_model_grad(ctx, torch.from_numpy(feat).cuda(), torch.from_numpy(target).cuda())
        ctx.sync()
        grad, loss = grad.cpu().numpy().astype(np.float64), float(loss.item())
    want_l, want_g = bm.loss_and_grad(params, feat, target)
    want_g = np.asarray(want_g, np.float64)
    assert abs(loss - float(want_l)) <= 1e-3 * float(want_l)
    lo = 0
    for name, size in SIZES:
        g, w = grad[lo:lo + size], want_g[lo:lo + size]
        lo += size
        assert np.linalg.norm(g - w) <= 2e-3 * np.linalg.norm(w), name
    assert lo == grad.size
