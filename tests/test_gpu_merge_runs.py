"""The center-star merge reads a CIGAR 32 characters at a time and takes its
runs side by side: alignments whose numbers and operations fall on every side
of those borders, long and many insertions in one place, split runs, exact
against the CPU merge."""
import numpy as np
import pytest

import seqgen
from oracle import center_star as cs

pytestmark = pytest.mark.gpu


def _random_ops(rs, C, gap_every, long):
    ops, p = [], 0
    while p < C:
        r = int(rs.integers(1, gap_every + 1, 1)[0])
        r = min(r, C - p)
        ops.append("=" * r if r % 2 else "X" * r)
        p += r
        g = int(rs.integers(0, long + 1, 1)[0])
        if g % 3 == 0 and p + g <= C:
            ops.append("D" * g)
            p += g
        else:
            ops.append("I" * g)
    return "".join(ops)


def _text(ops, split):
    out, k = [], 0
    while k < len(ops):
        e = k
        while e < len(ops) and ops[e] == ops[k] and (not split or e - k < split):
            e += 1
        out.append(f"{e - k}{ops[k]}")
        k = e
    return "".join(out)


@pytest.mark.parametrize("C,gap_every,long,split", [(1, 1, 5, 0), (40, 2, 3, 0), (300, 3, 2, 1), (300, 40, 130, 7),
                                                    (700, 1, 1, 0), (900, 12, 12, 0)])
def test_merge_of_given_alignments(C, gap_every, long, split):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(700 + C + long)
    center = rs.bases(C)
    seqs, ops = [center], ["=" * C]
    for _ in range(9):
        o = _random_ops(rs, C, gap_every, long)
        seqs.append(rs.bases(sum(c != "D" for c in o)))
        ops.append(o)
    texts = [_text(o, split) for o in ops]
    pool, off, lens = nw.pool_of(seqs)
    coff = np.concatenate([[0], np.cumsum([len(t) + 1 for t in texts])]).astype(np.uint64)
    cpool = np.frombuffer("".join(t + "\0" for t in texts).encode(), np.uint8).copy()
    clen = np.array([len(t) for t in texts], np.uint64)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        cols = nw.nw_msa_merge(ctx, pool, off, lens, 0, cpool, coff, clen)
        msa = np.zeros((len(seqs), cols + 1), np.uint8)
        assert nw.nw_msa_merge(ctx, pool, off, lens, 0, cpool, coff, clen, msa, cols + 1) == cols
    assert [r[:cols].tobytes().decode() for r in msa] == cs.merge(seqs, 0, ops)
