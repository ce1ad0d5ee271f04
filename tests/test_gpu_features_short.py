"""Features of short pairs, whose windows count their matches one by one, against
the CPU reference on both sides of the rule (windows of 255 and 257 offsets: the
longer sequence of 1,023 and 1,024 bases), with windows of fewer offsets than
bins, and with one letter, where every position matches.  The counts are whole
numbers; a feature is log1p of one over log1p of another: 1e-6 absolute."""
import numpy as np
import pytest

from oracle import band_model as bm

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4), (8, 7), (50, 61), (96, 103), (150, 150), (255, 300), (511, 200), (700, 1000), (1016, 1016),
          (1023, 1023), (1023, 600), (1024, 1024), (600, 1024), (1030, 1039)]


@pytest.mark.parametrize("letters", [4, 2, 1])
def test_features_of_short_windows(letters):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = np.random.default_rng(17)
    pairs = [(rs.integers(0, letters, m).astype(np.uint8), rs.integers(0, letters, n).astype(np.uint8))
             for m, n in SHAPES]
    pool, off, ln = nw.pool_of([s for p in pairs for s in p])
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        f = nw.nw_band_features(ctx, torch.from_numpy(pool).cuda(), off[0::2], ln[0::2], off[1::2], ln[1::2]).cpu().numpy()
    for k, (a, b) in enumerate(pairs):
        assert np.allclose(f[k], bm.features(a, b), rtol=0, atol=1e-6), (a.size, b.size)
