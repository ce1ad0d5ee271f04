"""Local and affine alignment keep a stripe's state every 128 steps and replay
the tiles a path crosses.  Exact against the oracle where that can go wrong:
lengths at and around the stripe and tile sizes, paths with long gaps across
tiles, end cells reached by several cells and chunks of one lane (ties), and
scores whose gaps cost nothing; and end cells under a budget too small for
all stripe rows."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu

ROWS = (255, 256, 257, 513)
COLS = (95, 96, 97, 98, 128, 129, 225, 1000)


def _pairs(seed):
    rs = seqgen.Stream(seed)
    out = []
    for m in ROWS:
        for n in COLS:
            b = rs.bases(max(m, n))
            a = b.copy()
            cut = int(rs.integers(1, max(m, n) - 1, 1)[0])
            a = np.concatenate([a[:cut], rs.bases(37), a[cut:]])[:m]  # a long gap across tiles
            out.append((a.astype(np.uint8), seqgen.mutate_distinct(b[:n], rs, 0.05, indel_mean=3.0)[0]))
    # the same word over and over: the largest H is reached in many cells
    unit = rs.bases(7)
    out.append((np.tile(unit, 60), np.concatenate([np.tile(unit, 5), 3 - np.tile(unit, 30), np.tile(unit, 5)])))
    out.append((np.tile(rs.bases(1), 300), np.concatenate([rs.bases(40), np.tile(unit[:1], 40), rs.bases(200)])))
    return out


def _pool(pairs):
    import paper_2412_21103_gb300 as nw
    pool, off, lens = nw.pool_of([s for p in pairs for s in p])
    return pool, off[0::2], lens[0::2], off[1::2], lens[1::2]


@pytest.mark.parametrize("sc", [(1, -1, -1), (2, -3, 0), (1, -1, 0)])
def test_local_tiles_and_ties(sc):
    import torch
    import paper_2412_21103_gb300 as nw
    pairs = _pairs(31)
    want = oracle.local_align_many(pairs, *sc)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        s, e, c = nw.nw_local_align_batch(ctx, *_pool(pairs), sc, nw.NW_CIGAR)
        s2, e2, _ = nw.nw_local_align_batch(ctx, *_pool(pairs), sc, 0)
    for k, (v, ends, ops) in enumerate(want):
        assert int(s[k]) == int(s2[k]) == v, k
        assert tuple(int(x) for x in e[k]) == tuple(ends) and c[k] == oracle.rle(ops), k
        assert tuple(int(x) for x in e2[k][2:]) == tuple(ends)[2:], k


def test_local_end_cells_with_two_rows_kept():
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(32)
    b = rs.bases(6000)
    pairs = [(seqgen.mutate_distinct(b[:5200], rs, 0.1, indel_mean=3.0)[0], b), (rs.bases(700), rs.bases(900))]
    want = oracle.local_align_many(pairs)
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=192 << 10) as ctx:
        s, e, _ = nw.nw_local_align_batch(ctx, *_pool(pairs), (1, -1, -1), 0)
    for k, (v, ends, _ops) in enumerate(want):
        assert int(s[k]) == v and tuple(int(x) for x in e[k][2:]) == tuple(ends)[2:], k


@pytest.mark.parametrize("sc", [(2, -3, -5, -2), (1, -1, 0, -1), (1, -1, -3, 0)])
def test_affine_tiles(sc):
    import torch
    import paper_2412_21103_gb300 as nw
    pairs = _pairs(33)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        s, c = nw.nw_affine_align_batch(ctx, *_pool(pairs), sc, nw.NW_CIGAR)
    for k, (v, ops) in enumerate(oracle.affine_align_many(pairs, *sc)):
        assert int(s[k]) == v and c[k] == oracle.rle(ops), k
