"""CIGAR assembly from moves (16 moves a thread as bit masks), exact against
the oracle: move counts around a thread's 16, a warp's and a CTA's moves, gaps
and mismatches at the threads' edges, one run over several chunks, few pairs
and many, one short pair (the CTA sizes), 'M' CIGARs."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 15, 16, 17, 31, 33, 511, 512, 513, 4095, 4096, 4097, 5000]


def _pairs(seed, sizes):
    rs = seqgen.Stream(seed)
    out = []
    for L in sizes:
        a = rs.bases(L)
        b = a.copy()
        for p in range(15, L, 16):  # mismatches on both sides of a thread's last move
            b[p] = (b[p] + 1) % 4 if p % 3 else b[p]
            if p + 1 < L and p % 5 == 0:
                b[p + 1] = (b[p + 1] + 2) % 4
        out += [(a, a.copy()), (a, b), (a, np.delete(b, range(min(14, L - 1), min(20, L))))]
    return out


def _check(ctx, pairs, flags):
    import paper_2412_21103_gb300 as nw
    pool, off, ln = nw.pool_of([s for p in pairs for s in p])
    s, c = nw.nw_align_batch(ctx, pool, off[0::2], ln[0::2], off[1::2], ln[1::2], (1, -1, -1), nw.NW_CIGAR | flags)
    for k, (v, ops) in enumerate(oracle.align_many(pairs)):
        want = oracle.rle(ops.replace("=", "M").replace("X", "M") if flags & nw.NW_CIGAR_M else ops)
        assert s[k] == v and c[k] == want, (k, pairs[k][0].size)


@pytest.mark.parametrize("m_flag", [False, True])
def test_few_and_many_pairs(m_flag):
    import torch
    import paper_2412_21103_gb300 as nw
    flags = nw.NW_CIGAR_M if m_flag else 0
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        _check(ctx, _pairs(61, SIZES), flags)                    # fewer pairs than SMs
        _check(ctx, _pairs(62, SIZES[:9] * 8), flags)            # more


@pytest.mark.parametrize("n", [3, 300, 1023, 1024, 2048, 16383, 16384, 16385, 40000])
def test_one_pair_over_chunks(n):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(63 + n)
    a = rs.bases(n)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        for b in (a.copy(), np.delete(a, range(n // 2, n // 2 + 2)), seqgen.mutate_distinct(a, rs, 0.1)[0]):
            s, c = nw.nw_align(ctx, nw.pack_codes(a), a.size, nw.pack_codes(b), b.size, (1, -1, -1), nw.NW_CIGAR)
            v, ops = oracle.align(a, b)
            assert s == v and c == oracle.rle(ops)
