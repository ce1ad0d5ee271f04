"""The band network's kernels at batches around a tile of samples and a share
of the weight gradients: outputs and gradients against the float64 reference
with the same BF16 roundings.  Tolerances: an FP32 sum of at most 128 products
per unit (relative error about 128 * 2^-24 = 8e-6) can turn the BF16 rounding of
an activation here and there, which changes it by 2^-8 of itself, a gradient
(a product of an error and an activation) by twice that, and an output by far
less than 1e-2 of its magnitude: 1e-2 of the largest gradient or output."""
import numpy as np
import pytest

import seqgen
from oracle import band_model as bm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 32, 33, 65, 257, 1031])
def test_outputs_and_gradients(n):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(61 + n)
    feat = rs.uniform(n * 65).reshape(n, 65).astype(np.float32)
    target = (3.0 + 4.0 * rs.uniform(n)).astype(np.float32)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        nw.nw_band_model_init(ctx, 5)
        params = nw.nw_band_model_get(ctx)
        x, t = torch.from_numpy(feat).cuda(), torch.from_numpy(target).cuda()
        y = nw.nw_band_model_forward(ctx, x).cpu().numpy()
        grad, loss = nw.nw_band_model_grad(ctx, x, t)
        ctx.sync()
        grad, loss = grad.cpu().numpy(), float(loss.item())
    want_y = np.asarray(bm.forward(params, feat)[0]).reshape(n)
    assert np.abs(y - want_y).max() <= 1e-2 * max(1.0, np.abs(want_y).max())
    want_l, want_g = bm.loss_and_grad(params, feat, target)
    assert abs(loss - float(want_l)) <= 2e-2 * max(1.0, float(want_l))
    assert np.abs(grad - np.asarray(want_g)).max() <= 1e-2 * np.abs(want_g).max()
