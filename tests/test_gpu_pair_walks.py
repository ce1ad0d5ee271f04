"""Pairs of a batch on the single-pair kernel run longest chain first, but are
walked by their moves: above 16,384 in linked pieces, else by runs.  A tall
pair of 16,384 moves has the longer chain, a wide one of 16,400 the longer
walk, which must be cut into pieces whatever stands before it."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,pieces", [([(9000, 7384), (7300, 9100)], True), ([(9000, 7384), (7300, 9000)], False)])
def test_long_walks_behind_a_tall_pair(sizes, pieces):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(88)
    pairs = []
    for m, n in sizes:
        b = rs.bases(max(m, n) + 400)
        pairs.append((seqgen.mutate_distinct(b, rs, 0.1, indel_mean=3.0)[0][:m], b[:n]))
        assert pairs[-1][0].size == m
    pool, off, lens = nw.pool_of([s for p in pairs for s in p])
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        ctx.set_profiling(True)
        s, c = nw.nw_align_batch(ctx, pool, off[0::2], lens[0::2], off[1::2], lens[1::2], (1, -1, -1), nw.NW_CIGAR)
        stats = ctx.kernel_stats()
    assert stats["bpair_fill_ptr"][0] == 1 and stats["tb_runs"][0] == 1
    assert ("tb_spec" in stats) == pieces
    for k, (v, ops) in enumerate(oracle.align_many(pairs)):
        assert s[k] == v and c[k] == oracle.rle(ops), k
