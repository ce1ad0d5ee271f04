"""Affine walks take a gap a run at a time: gaps of either kind shorter and longer
than a warp's 32 lanes, than a tile of 128 steps and than the three tiles
replayed at once, across stripes, up to the first row and column, and with free
extensions (where ties close the gap), against the oracle."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


def _pairs():
    rs = seqgen.Stream(630)
    out = []
    for gap in (1, 31, 32, 33, 64, 127, 128, 129, 380, 400, 900):
        for left in (0, 5, 250):
            a = rs.bases(left + 60)
            b = np.concatenate([a[:left], rs.bases(gap), a[left:]]).astype(np.uint8)
            out += [(a, b), (b, a)]
    out += [(rs.bases(150), rs.bases(1000)), (rs.bases(1000), rs.bases(150)), (rs.bases(1), rs.bases(700)),
            (rs.bases(700), rs.bases(1))]
    return out


@pytest.mark.parametrize("sc", [(2, -3, -5, -2), (1, -1, -3, 0), (1, -1, 0, -1), (2, -2, -1, 0)])
def test_long_gaps(sc):
    import torch
    import paper_2412_21103_gb300 as nw
    pairs = _pairs()
    pool, off, ln = nw.pool_of([s for p in pairs for s in p])
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        s, c = nw.nw_affine_align_batch(ctx, pool, off[0::2], ln[0::2], off[1::2], ln[1::2], sc, nw.NW_CIGAR)
    for k, (v, ops) in enumerate(oracle.affine_align_many(pairs, *sc)):
        assert int(s[k]) == v and c[k] == oracle.rle(ops), k
