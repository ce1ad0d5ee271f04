"""The measured peak of the bit-sliced update bounds the score kernel that it
is the roofline of: all-vs-all of 512 sequences, cells of the grids over the
kernel's own time."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_the_score_kernel_stays_below_its_peak():
    import torch
    import paper_2412_21103_gb300 as nw
    rng = np.random.default_rng(3)
    ln = rng.integers(500, 1501, 512).astype(np.uint32)
    off = (np.arange(512) * 400).astype(np.uint64)
    pool = torch.from_numpy(rng.integers(0, 256, 512 * 400, dtype=np.uint8)).cuda()
    out = torch.zeros((512, 512), dtype=torch.int32, device="cuda")
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        peak = nw.nw_peak_int(ctx, 11, 1 << 12) * 1e9
        for _ in range(3):
            nw.nw_score_all_pairs(ctx, pool, off, ln, (1, -1, -1), 0, out)
        ctx.sync()
        ctx.set_profiling(True)
        for _ in range(5):
            nw.nw_score_all_pairs(ctx, pool, off, ln, (1, -1, -1), 0, out)
        n, ms = ctx.kernel_stats()["bits_score"]
    x = ln.astype(np.float64)
    cells = (x.sum() ** 2 - (x * x).sum()) / 2
    assert 0.3 * peak < cells / (ms / n * 1e-3) < peak
