"""The window band's walk recomputes the pointers of a block of anti-diagonals
in a sub-window around the path.  Exact against the oracle where that can go
wrong: pairs whose last anti-diagonal lies at, just before and just after a
block's end, windows of fewer, as many and more words than the sub-window,
paths that drift across a block by long gaps, and
walks split into stretches that join or do not."""
import os

import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,stretch", [(3, None), (200, None), (250, None), (600, None), (3, 1), (100, 1), (200, 2),
                                       (300, 7), (600, 3)])
def test_blocks_windows_and_drift(w, stretch, monkeypatch):
    if stretch:
        # blocks of a stretch: with one or two the ways between them often miss
        # the next stretch, and the pair is walked as a whole
        monkeypatch.setenv("NW_BBAND_STRETCH", str(stretch))
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(7100 + w)
    pairs = []
    for base in (1152, 2304):  # multiples of the block lengths in use
        for extra in (-1, 0, 1, 63, 64, 65):
            m = (base + extra) // 2 + 2 * w
            a = rs.bases(m)
            gap = min(w, 180)  # gaps as long as a band of this width certifies
            p = int(rs.integers(m // 4, m // 2, 1)[0])
            q = int(rs.integers(m // 2, 3 * m // 4, 1)[0])
            b = np.concatenate([a[:p], rs.bases(gap // 2), a[p:q], a[q + gap // 2:]])
            b = np.concatenate([b, rs.bases(1)]) if (m + b.size + base + extra) % 2 else b
            pairs.append((a, b.astype(np.uint8)))
            pairs.append((a, seqgen.mutate_distinct(a, rs, 0.05, indel_frac=0.4, indel_mean=3.0)[0]))
    pool, off, lens = nw.pool_of([s for p in pairs for s in p])
    os.environ["NW_BAND_KEEP"] = "1"  # every pair stays in the banded rounds
    try:
        with nw.Context(0, torch.cuda.current_stream()) as ctx:
            scores, cigars = nw.nw_align_batch_banded(ctx, pool, off[0::2], lens[0::2], off[1::2], lens[1::2],
                                                      np.full(len(pairs), w, np.uint32), (1, -1, -1), nw.NW_CIGAR)
            assert sum(nw.nw_ctx_band_stats(ctx)["certified_round"]) >= len(pairs) // 2
    finally:
        del os.environ["NW_BAND_KEEP"]
    for k, (s, ops) in enumerate(oracle.align_many(pairs, 1, -1, -1)):
        assert scores[k] == s, k
        assert cigars[k] == oracle.rle(ops), k
