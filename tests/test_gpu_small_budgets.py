"""Calls on contexts whose scratch budget leaves little beyond what the call
cannot do without: the plan falls back to the form that fits instead of
reporting NW_ERR_OOM, with the results of a context of any size.  Sequences are
random bytes of a device pool (four bases each)."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


def _bases(pool, off, n):
    b = pool[off:off + (n + 3) // 4]
    return ((b[:, None] >> (2 * np.arange(4, dtype=np.uint8))) & 3).reshape(-1)[:n].astype(np.uint8)


def _random_pool(seed, nbytes):
    return np.random.default_rng(seed).integers(0, 256, nbytes, dtype=np.uint8)


def _scores(nw, ctx, pool, a, m, b, n, sc):
    import torch
    out = torch.full((len(m),), -1, dtype=torch.int32, device="cuda")
    nw.nw_align_batch(ctx, pool, a, m, b, n, sc, 0, scores=out)
    ctx.sync()
    return out.cpu().numpy()


# few sequences far up in a large pool, read by many pairs: slots of the pairs'
# own would take 3.9 MB (first) or, fitting by themselves, leave too little
# for the row buffers (second)
@pytest.mark.parametrize("m,n,pairs,budget", [(1500, 1500, 5000, 3 << 20), (60, 20000, 32, 1400 << 10)])
def test_score_batch_of_few_sequences_in_a_large_pool(m, n, pairs, budget):
    import torch
    import paper_2412_21103_gb300 as nw
    pool = _random_pool(5, 8 << 20)
    at = pool.size - 8192
    a = np.full(pairs, at, np.uint64)
    b = np.full(pairs, at + 1024, np.uint64)
    ml, nl = np.full(pairs, m, np.uint32), np.full(pairs, n, np.uint32)
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=budget) as ctx:
        got = _scores(nw, ctx, torch.from_numpy(pool).cuda(), a, ml, b, nl, (1, -1, -1))
    assert (got == oracle.score(_bases(pool, at, m), _bases(pool, at + 1024, n))).all()


def test_score_batch_in_units_without_room_for_its_planes():
    """60,000 pairs of 1,000 bases scored +2/-1/-2: 45 MB on the bit planes, 24
    MB on the scalar kernel."""
    import torch
    import paper_2412_21103_gb300 as nw
    count, n = 60000, 1000
    pool = _random_pool(6, 2 * count * 250)
    off = np.arange(2 * count, dtype=np.uint64) * 250
    ln = np.full(count, n, np.uint32)
    dev = torch.from_numpy(pool).cuda()
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        want = _scores(nw, ctx, dev, off[0::2], ln, off[1::2], ln, (2, -1, -2))
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=30 << 20) as ctx:
        got = _scores(nw, ctx, dev, off[0::2], ln, off[1::2], ln, (2, -1, -2))
    assert (got == want).all()
    for k in (0, 31, count - 1):
        assert got[k] == oracle.score(_bases(pool, int(off[2 * k]), n), _bases(pool, int(off[2 * k + 1]), n), 2, -1, -2)


def _similar(rs, n, subs):
    """A sequence of n bases and a copy with `subs` substitutions."""
    a = rs.bases(n)
    b = a.copy()
    at = rs.integers(0, n - 1, subs)
    b[at] = (b[at] + 1 + rs.integers(0, 2, subs)) % 4
    return a, b.astype(np.uint8)


def _banded(nw, ctx, pairs, w, sc=(1, -1, -1)):
    """Banded alignments on device buffers: scores, CIGARs, pairs certified in a band."""
    import torch
    pool, off, ln = nw.pool_of([s for p in pairs for s in p])
    co = np.concatenate([[0], np.cumsum([nw.nw_cigar_bound(a.size, b.size) for a, b in pairs])]).astype(np.uint64)
    s = torch.full((len(pairs),), -1, dtype=torch.int32, device="cuda")
    cp = torch.zeros(int(co[-1]), dtype=torch.uint8, device="cuda")
    cl = torch.zeros(len(pairs), dtype=torch.int64, device="cuda")
    before = sum(nw.nw_ctx_band_stats(ctx)["certified_round"])
    nw.nw_align_batch_banded(ctx, torch.from_numpy(pool).cuda(), off[0::2], ln[0::2], off[1::2], ln[1::2],
                             np.full(len(pairs), w, np.uint32), sc, nw.NW_CIGAR, s, cp, co, cl)
    ctx.sync()
    h, n = cp.cpu().numpy(), cl.cpu().numpy()
    text = [bytes(h[int(co[k]):int(co[k]) + int(n[k])]).decode() for k in range(len(pairs))]
    return s.cpu().numpy(), text, sum(nw.nw_ctx_band_stats(ctx)["certified_round"]) - before


def _align(nw, ctx, pairs, sc=(1, -1, -1)):
    import torch
    pool, off, ln = nw.pool_of([s for p in pairs for s in p])
    co = np.concatenate([[0], np.cumsum([nw.nw_cigar_bound(a.size, b.size) for a, b in pairs])]).astype(np.uint64)
    s = torch.full((len(pairs),), -1, dtype=torch.int32, device="cuda")
    cp = torch.zeros(int(co[-1]), dtype=torch.uint8, device="cuda")
    cl = torch.zeros(len(pairs), dtype=torch.int64, device="cuda")
    nw.nw_align_batch(ctx, torch.from_numpy(pool).cuda(), off[0::2], ln[0::2], off[1::2], ln[1::2], sc,
                      nw.NW_CIGAR, s, cp, co, cl)
    ctx.sync()
    h, n = cp.cpu().numpy(), cl.cpu().numpy()
    return s.cpu().numpy(), [bytes(h[int(co[k]):int(co[k]) + int(n[k])]).decode() for k in range(len(pairs))]


@pytest.mark.parametrize("sc", [(1, -1, -1), (2, -1, -2)])
def test_band_after_a_batch_that_filled_the_scratch(sc, monkeypatch):
    """Alignments of 3 kb leave records of half the budget behind; the pairs of
    the next call still run in their band (+2/-1/-2: on the scalar banded kernel,
    whose pointer words fit only once the records are handed back)."""
    import torch
    import paper_2412_21103_gb300 as nw
    monkeypatch.setenv("NW_BAND_KEEP", "1")
    rs = seqgen.Stream(91)
    first = [_similar(rs, 3000, 90) for _ in range(200)]
    pairs = [_similar(rs, 8000, 200) for _ in range(3)]
    want = oracle.align_many(pairs, *sc)
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=16 << 20) as ctx:
        _align(nw, ctx, first, sc)
        s, c, banded = _banded(nw, ctx, pairs, 900, sc)
    assert banded == len(pairs)
    assert list(s) == [v for v, _ in want] and c == [oracle.rle(o) for _, o in want]


def test_band_of_a_pair_whose_full_records_do_not_fit(monkeypatch):
    """A band of 5.6 million cells under 2 MB: kept planes take 24 KB of it."""
    import torch
    import paper_2412_21103_gb300 as nw
    monkeypatch.setenv("NW_BAND_KEEP", "1")
    pairs = [_similar(seqgen.Stream(92), 6000, 180)]
    want = oracle.align_many(pairs)
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=2 << 20) as ctx:
        s, c, banded = _banded(nw, ctx, pairs, 200)
    assert banded == 1
    assert list(s) == [v for v, _ in want] and c == [oracle.rle(o) for _, o in want]


def test_band_waves_leave_room_for_the_moves(monkeypatch):
    """Narrow bands keep fewer bytes of planes than their walks have moves: 600
    pairs of 5 kb keep 1.5 MB and walk 6 MB, under a budget of 5."""
    import torch
    import paper_2412_21103_gb300 as nw
    monkeypatch.setenv("NW_BAND_KEEP", "1")
    rs = seqgen.Stream(93)
    pairs = [_similar(rs, 5000, 10) for _ in range(600)]
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=5 << 20) as ctx:
        s, c, banded = _banded(nw, ctx, pairs, 20)
    assert banded == len(pairs)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        s2, c2 = _align(nw, ctx, pairs)
    assert (s == s2).all() and c == c2
    for k in (0, 299, 599):
        v, ops = oracle.align(*pairs[k])
        assert s[k] == v and c[k] == oracle.rle(ops)


@pytest.mark.parametrize("kind", ["local", "affine"])
def test_waves_of_short_pairs_count_their_moves_and_tables(kind):
    """20,000 pairs of 90 bases keep no state between steps, but have 8 MB of
    moves and tables, under a budget of 4."""
    import torch
    import paper_2412_21103_gb300 as nw
    count, n = 20000, 90
    pool = _random_pool(7, 2 * count * 23)
    off = np.arange(2 * count, dtype=np.uint64) * 23
    ln = np.full(count, n, np.uint32)
    dev = torch.from_numpy(pool).cuda()
    co = np.arange(count + 1, dtype=np.uint64) * nw.nw_cigar_bound(n, n)
    got = []
    for budget in (4 << 20, 0):
        with nw.Context(0, torch.cuda.current_stream(), mem_budget=budget) as ctx:
            s = torch.full((count,), -1, dtype=torch.int32, device="cuda")
            e = torch.zeros((count, 4), dtype=torch.int32, device="cuda")
            cp = torch.zeros(int(co[-1]), dtype=torch.uint8, device="cuda")
            cl = torch.zeros(count, dtype=torch.int64, device="cuda")
            if kind == "local":
                nw.nw_local_align_batch(ctx, dev, off[0::2], ln, off[1::2], ln, (1, -1, -1), nw.NW_CIGAR, s, e, cp, co, cl)
            else:
                nw.nw_affine_align_batch(ctx, dev, off[0::2], ln, off[1::2], ln, (2, -3, -5, -2), nw.NW_CIGAR, s, cp, co, cl)
            ctx.sync()
            got.append([x.cpu().numpy() for x in (s, e, cl, cp)])
    for x, y in zip(got[0][:3], got[1][:3]):
        assert (x == y).all()
    texts = [[bytes(g[3][int(co[k]):int(co[k]) + int(g[2][k])]) for k in range(count)] for g in got]
    assert texts[0] == texts[1]
    for k in (0, 7777, count - 1):
        pair = (_bases(pool, int(off[2 * k]), n), _bases(pool, int(off[2 * k + 1]), n))
        if kind == "local":
            v, ends, ops = oracle.local_align_many([pair])[0]
            assert tuple(int(x) for x in got[0][1][k]) == tuple(ends)
        else:
            v, ops = oracle.affine_align_many([pair], 2, -3, -5, -2)[0]
        assert int(got[0][0][k]) == v and texts[0][k].decode() == oracle.rle(ops)


def test_alignments_whose_planar_copies_alone_fill_the_budget():
    """1,500 pairs of 1 kb: .8 MB of planar copies, .3 to .5 MB of records a pair,
    under a budget of 1.2 MB."""
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(94)
    pairs = [_similar(rs, 1000, 40) for _ in range(1500)]
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=1200 << 10) as ctx:
        s, c = _align(nw, ctx, pairs)
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        s2, c2 = _align(nw, ctx, pairs)
    assert (s == s2).all() and c == c2
    for k in (0, 700, 1499):
        v, ops = oracle.align(*pairs[k])
        assert s[k] == v and c[k] == oracle.rle(ops)


# budgets that the scalar kernel fits, a warp's records and planar copies of some
# pairs do not; twice, because the second call finds the first one's slots
@pytest.mark.parametrize("rows,cols,count,budget", [((2000, 4000), (2000, 4000), 4, 1680000), ((300, 1500), (300, 1500), 200, 497000),
                                                    ((100, 300), (5000, 20000), 50, 3780000),
                                                    ((5000, 20000), (100, 300), 50, 1680000)])
@pytest.mark.parametrize("sc", [(1, -1, -1), (2, -1, -2)])
def test_alignments_that_fit_only_the_scalar_kernel(rows, cols, count, budget, sc):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(96)
    pairs = [(rs.bases(int(m)), rs.bases(int(n))) for m, n in zip(rs.integers(*rows, count), rs.integers(*cols, count))]
    with nw.Context(0, torch.cuda.current_stream(), mem_budget=budget) as ctx:
        got = [_align(nw, ctx, pairs, sc) for _ in range(2)]
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        s, c = _align(nw, ctx, pairs, sc)
    for s2, c2 in got:
        assert (s == s2).all() and c == c2
    v, ops = oracle.align(*pairs[0], *sc)
    assert s[0] == v and c[0] == oracle.rle(ops)
