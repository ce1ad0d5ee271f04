"""The local fill with few stripe jobs takes its scores from byte permutes, with
more than 12 per SM from shared memory: the same pairs -- rows and columns around
stripes and tiles, rows past the end, ragged last chunks -- once and repeated
until they are that many, against the oracle."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


def _pairs():
    rs = seqgen.Stream(620)
    out = []
    for m in (1, 7, 8, 9, 255, 256, 257, 513):
        for n in (1, 31, 32, 33, 64, 97, 129, 700):
            b = rs.bases(max(m, n) + 80)
            out.append((seqgen.mutate_distinct(b, rs, 0.1, indel_mean=3.0)[0][:m], b[:n]))
    return out


@pytest.mark.parametrize("sc", [(1, -1, -1), (40, -40, -3), (5, -4, 0)])
def test_scores_from_permutes_and_from_the_table(sc):
    import torch
    import paper_2412_21103_gb300 as nw
    pairs = _pairs()
    want = oracle.local_align_many(pairs, *sc)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for times in (1, 12 * sms // len(pairs) + 1):
        pool, off, ln = nw.pool_of([s for p in pairs for s in p])
        ao, al, bo, bl = (np.tile(x, times) for x in (off[0::2], ln[0::2], off[1::2], ln[1::2]))
        with nw.Context(0, torch.cuda.current_stream()) as ctx:
            s, e, c = nw.nw_local_align_batch(ctx, pool, ao, al, bo, bl, sc, nw.NW_CIGAR)
            s2, e2, _ = nw.nw_local_align_batch(ctx, pool, ao, al, bo, bl, sc, 0)
        for k in range(len(s)):
            v, ends, ops = want[k % len(pairs)]
            assert int(s[k]) == int(s2[k]) == v, k
            assert tuple(int(x) for x in e[k]) == tuple(ends) and c[k] == oracle.rle(ops), k
            assert tuple(int(x) for x in e2[k][2:]) == tuple(ends)[2:], k
