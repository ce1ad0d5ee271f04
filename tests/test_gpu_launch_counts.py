"""Kernel counts of the statistics: the window walk is one launch for whole
pairs and seven in stretches (first cells, stretches, ways between them, and
twice linking and walking what did not join)."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretch,launches", [(None, 7), ("100000", 1)])
def test_window_walk(stretch, launches, monkeypatch):
    import torch
    import paper_2412_21103_gb300 as nw
    monkeypatch.setenv("NW_BAND_KEEP", "1")
    if stretch:
        monkeypatch.setenv("NW_BBAND_STRETCH", stretch)
    rs = seqgen.Stream(95)
    a = rs.bases(6000)  # 188 blocks: three stretches of 72
    b = seqgen.mutate_distinct(a, rs, 0.03)[0]
    pool, off, ln = nw.pool_of([a, b])
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        ctx.set_profiling(True)
        s, c = nw.nw_align_batch_banded(ctx, pool, off[0::2], ln[0::2], off[1::2], ln[1::2], np.array([300], np.uint32),
                                        (1, -1, -1), nw.NW_CIGAR)
        assert ctx.kernel_stats()["bband_walk"][0] == launches
    v, ops = oracle.align(a, b)
    assert s[0] == v and c[0] == oracle.rle(ops)
