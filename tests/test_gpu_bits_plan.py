"""Launch plans of the bit-sliced score kernel: all-vs-all jobs named by class
(rows of equal stripe count) and batches whose sequences get slots of their
own or, when they are read several times over, one slot each.  Lengths at the
edges of stripes and chunks, empty sequences and classes of every size,
against the oracle."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 2, 31, 32, 33, 63, 64, 65, 66, 95, 96, 97, 128, 129, 200]


def _seqs(seed, lens):
    rs = seqgen.Stream(seed)
    root = rs.bases(max(lens) + 1)
    return [seqgen.mutate_distinct(root[:n], rs, 0.2)[0][:n] if n else root[:0] for n in lens]


@pytest.mark.parametrize("lens", [EDGES, [64] * 40, [40] * 3 + [33] * 35 + [500], [0, 0, 5], [7]])
@pytest.mark.parametrize("sc", [(1, -1, -1), (1, 0, -1)])
def test_all_pairs_classes(lens, sc):
    import torch
    import paper_2412_21103_gb300 as nw
    seqs = _seqs(41, lens)
    pool, off, ln = nw.pool_of(seqs)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        got = nw.nw_score_all_pairs(ctx, pool, off, ln, sc)
    for i in range(len(seqs)):
        for j in range(len(seqs)):
            want = sc[0] * len(seqs[i]) if i == j else oracle.score(seqs[min(i, j)], seqs[max(i, j)], *sc)
            assert got[i, j] == want, (i, j)


@pytest.mark.parametrize("repeated", [False, True])
def test_batch_slots(repeated):
    import torch
    import paper_2412_21103_gb300 as nw
    seqs = _seqs(42, EDGES + [150] * 20)
    n = len(seqs)
    pairs = [(i, j) for i in range(n) for j in range(n)] if repeated else [(i, n - 1 - i) for i in range(n)]
    pool, off, ln = nw.pool_of(seqs)
    a, b = np.array([p[0] for p in pairs]), np.array([p[1] for p in pairs])
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        got, _ = nw.nw_align_batch(ctx, pool, off[a], ln[a], off[b], ln[b], (1, -1, -1), 0)
    for k, (i, j) in enumerate(pairs):
        assert got[k] == oracle.score(seqs[i], seqs[j], 1, -1, -1), (i, j)


@pytest.mark.parametrize("words", [1, 2, 4])
@pytest.mark.parametrize("sc", [(1, -1, -1), (1, 0, -1)])
def test_words_per_lane(words, sc, monkeypatch):
    """Every number of words a lane on rows around multiples of its stripes and
    columns around its shortest period, lanes of one warp differing in both."""
    import torch
    import paper_2412_21103_gb300 as nw
    monkeypatch.setenv("NW_BITS_WORDS", str(words))
    h = 32 * words
    rows = [1, 2, h - 1, h, h + 1, 2 * h - 3, 2 * h, 3 * h - 31, 5 * h + 1]
    cols = [1, 3, 31, 32, 33, 65, 32 * (words + 2), 32 * (words + 3), 32 * (words + 3) + 1, 32 * (words + 5) - 1, 700]
    rs = seqgen.Stream(43)
    root = rs.bases(800)
    pairs = []
    for m in rows:
        for n in cols:
            a = root[:m]
            pairs.append((a, seqgen.mutate_distinct(root, rs, 0.2)[0][:n]))
    pool, off, ln = nw.pool_of([s for p in pairs for s in p])
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        got, _ = nw.nw_align_batch(ctx, pool, off[0::2], ln[0::2], off[1::2], ln[1::2], sc, 0)
    assert list(got) == oracle.score_many(pairs, *sc)
