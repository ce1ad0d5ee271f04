"""Features of the learned band, counted on bit planes 32 positions at a time,
against the CPU reference at the edges of words, windows, bins and anchors.
The counts are whole numbers; a feature is log1p of one over log1p of another,
each within a few units in the last place: 1e-6 absolute."""
import numpy as np
import pytest

from oracle import band_model as bm

pytestmark = pytest.mark.gpu


def _pool(pairs):
    import paper_2412_21103_gb300 as nw
    pool, off, lens = nw.pool_of([s for p in pairs for s in p])
    return pool, off[0::2], lens[0::2], off[1::2], lens[1::2]


SHAPES = [(4, 4), (5, 4), (4, 300), (300, 4), (34, 35), (35, 36), (67, 66), (258, 259), (259, 260), (260, 97),
          (31, 1000), (1000, 31), (511, 515), (2051, 2048), (2000, 1100), (900, 2500)]


@pytest.mark.parametrize("letters", [4, 1])
def test_features_at_word_window_and_anchor_edges(letters):
    import torch

    import paper_2412_21103_gb300 as nw
    ctx = nw.Context(0, torch.cuda.current_stream())
    rs = np.random.default_rng(7)
    pairs = [(rs.integers(0, letters, m).astype(np.uint8), rs.integers(0, letters, n).astype(np.uint8))
             for m, n in SHAPES]
    pairs += [(np.zeros(0, np.uint8), np.zeros(9, np.uint8)), (np.zeros(3, np.uint8), np.zeros(40, np.uint8))]
    pool, ao, al, bo, bl = _pool(pairs)
    f = nw.nw_band_features(ctx, torch.from_numpy(pool).cuda(), ao, al, bo, bl).cpu().numpy()
    for k, (a, b) in enumerate(pairs):
        assert np.allclose(f[k], bm.features(a, b), rtol=0, atol=1e-6), (a.size, b.size)
    ctx.close()


def test_features_of_the_longest_accepted_b():
    """200,000 bases need more than the default shared memory; one match only."""
    import torch

    import paper_2412_21103_gb300 as nw
    ctx = nw.Context(0, torch.cuda.current_stream())
    a, b = np.zeros(5000, np.uint8), np.ones(200000, np.uint8)
    b[120000:120004] = 0
    pool, ao, al, bo, bl = _pool([(a, b)])
    f = nw.nw_band_features(ctx, torch.from_numpy(pool).cuda(), ao, al, bo, bl).cpu().numpy()[0]
    m, n, W = a.size, b.size, b.size // 8
    hist = np.zeros(64)
    for k in range(256):
        i = (k * (m - 4)) // 255
        c0 = i + int(round((n - m) * i / m))
        if abs(120000 - c0) <= W:
            hist[((120000 - c0 + W) * 64) // (2 * W + 1)] += 1
    assert np.allclose(f[:64], np.log1p(hist) / np.log1p(256), rtol=0, atol=1e-6)
    ctx.close()
