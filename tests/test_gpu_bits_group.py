"""CIGAR batches on groups of lanes of the bit-sliced kernel (k_bits_group) and
the walk by runs, against the oracle: rows at and around multiples of a bit
stripe (31), of a group's stripes and of a pass, columns at and around the
chunks of 32 steps (where a pass follows the one before without a gap), long
gaps, unrelated pairs, empty sides, two-plane scorings (as they are, and in
units of a common divisor), 'M' CIGARs, and a
budget that splits the batch into waves."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu

ROWS = [1, 30, 31, 32, 62, 63, 123, 124, 125, 249, 312, 993]
COLS = [1, 2, 31, 33, 34, 66, 98, 130, 162, 290, 1025]


def _pairs(seed, rows, cols):
    rs = seqgen.Stream(seed)
    out = []
    for m in rows:
        for n in cols:
            b = rs.bases(max(m, n) + 60)
            a = np.concatenate([b[:n // 2], b[n // 2 + 40:]])[:m] if (m + n) % 3 else rs.bases(m)
            out.append((a.astype(np.uint8), seqgen.mutate_distinct(b, rs, 0.1, indel_mean=3.0)[0][:n]))
    return out


def _check(ctx, pairs, sc, flags=0):
    import paper_2412_21103_gb300 as nw
    pool, off, lens = nw.pool_of([s for p in pairs for s in p])
    s, c = nw.nw_align_batch(ctx, pool, off[0::2], lens[0::2], off[1::2], lens[1::2], sc, nw.NW_CIGAR | flags)
    for k, (v, ops) in enumerate(oracle.align_many(pairs, *sc)):
        want = oracle.rle(ops.replace("=", "M").replace("X", "M") if flags & nw.NW_CIGAR_M else ops)
        assert s[k] == v and c[k] == want, (k, pairs[k][0].size, pairs[k][1].size)


@pytest.mark.parametrize("sc", [(1, -1, -1), (1, 0, -1), (1, -2, -1), (2, -1, -2), (2, -2, -2), (4, -2, -1)])
def test_shapes(sc):
    import torch
    import paper_2412_21103_gb300 as nw
    empty = np.zeros(0, np.uint8)
    pairs = _pairs(51, ROWS, COLS) + [(empty, empty), (empty, seqgen.Stream(1).bases(9)), (seqgen.Stream(2).bases(9), empty)]
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        ctx.set_profiling(True)
        _check(ctx, pairs, sc)
        assert ctx.kernel_stats()["bgroup_fill_ptr"][0] > 0
        _check(ctx, pairs[:40], sc, nw.NW_CIGAR_M)
        pool, off, lens = nw.pool_of([s for p in pairs for s in p])
        s, _ = nw.nw_align_batch(ctx, pool, off[0::2], lens[0::2], off[1::2], lens[1::2], sc, 0)
        assert list(s) == oracle.score_many(pairs, *sc)


@pytest.mark.parametrize("sc", [(2, -1, -2), (2, -2, -2)])
def test_score_batches_in_units(sc):
    """Enough short pairs to fill the GPU take the bit planes in units of the
    common divisor, a few the scalar kernel; the scores are the same."""
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(54)
    seqs = [rs.bases(int(n)) for n in rs.integers(20, 70, 24000)]
    pool, off, lens = nw.pool_of(seqs)
    want = oracle.score_many(list(zip(seqs[0::2], seqs[1::2])), *sc)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        ctx.set_profiling(True)
        for n, bits in ((12000, True), (30, sc[0] - 2 * sc[2] <= 3)):
            ctx.reset_stats()
            s, _ = nw.nw_align_batch(ctx, pool, off[0:2 * n:2], lens[0:2 * n:2], off[1:2 * n:2], lens[1:2 * n:2], sc, 0)
            assert list(s) == want[:n]
            assert (ctx.kernel_stats().get("bits_score", (0, 0.0))[0] > 0) == bits


def test_many_pairs_take_few_lanes_and_waves():
    import torch
    import paper_2412_21103_gb300 as nw
    pairs = _pairs(52, [300] * 20, [280, 310, 350] * 6)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        _check(ctx, pairs, (1, -1, -1))
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=8 << 20) as ctx:
        _check(ctx, pairs, (1, -1, -1))
