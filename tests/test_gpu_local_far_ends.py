"""End cells of pairs whose largest H comes again far on: reads against long
references with copies of the read (exact, or of its end only) planted many
tiles apart, so that the first cell in row-major order -- the smallest row, then
the smallest column -- may lie in any of them, before, in and after the last
full tile; pairs of one to five stripes, with and without kept states, and a
budget that keeps none."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


def _pairs():
    rs = seqgen.Stream(610)
    out = []
    for m, n in [(40, 3000), (200, 5000), (256, 4100), (300, 2500), (700, 1500), (1024, 1300), (1100, 1400)]:
        for copies in (1, 2, 5):
            a = rs.bases(m)
            b = rs.bases(n)
            w = min(m, 60)
            for c in range(copies):
                # the same stretch of the read again; its first rows in some, its last in others
                part = a[:w] if c % 2 else a[m - w:]
                at = (n - w) * c // max(copies - 1, 1) if copies > 1 else (n - w) // 2
                b[at:at + w] = part
            out.append((a, b.astype(np.uint8)))
    # every column alike: the largest H all along the last row
    out.append((np.zeros(30, np.uint8), np.zeros(1500, np.uint8)))
    out.append((np.zeros(250, np.uint8), np.concatenate([np.zeros(900, np.uint8), np.ones(400, np.uint8), np.zeros(900, np.uint8)])))
    return out


@pytest.mark.parametrize("budget", [0, 600 << 10])
@pytest.mark.parametrize("sc", [(1, -1, -1), (2, -3, -2), (1, -1, 0)])
def test_first_cell_among_far_copies(sc, budget):
    import torch
    import paper_2412_21103_gb300 as nw
    pairs = _pairs()
    pool, off, ln = nw.pool_of([s for p in pairs for s in p])
    args = (pool, off[0::2], ln[0::2], off[1::2], ln[1::2], sc)
    want = oracle.local_align_many(pairs, *sc)
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=budget) as ctx:
        s, e, _ = nw.nw_local_align_batch(ctx, *args, 0)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        s2, e2, c2 = nw.nw_local_align_batch(ctx, *args, nw.NW_CIGAR)
    for k, (v, ends, ops) in enumerate(want):
        assert int(s[k]) == int(s2[k]) == v, k
        assert tuple(int(x) for x in e[k][2:]) == tuple(ends)[2:], k
        assert tuple(int(x) for x in e2[k]) == tuple(ends) and c2[k] == oracle.rle(ops), k
