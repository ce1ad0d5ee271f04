"""Local alignment on a context that holds an unreported error: the fill's
waits give up early, so stripes stay undone, and the trace must follow none
of them.  The error is a bad base packed on the device, the call before it
leaves longer pairs' results in the scratch slots; the sync reports the bad
base and the next call is exact."""
import numpy as np
import pytest

import oracle
import seqgen

pytestmark = pytest.mark.gpu


def _call(nw, ctx, pairs, cigar):
    import torch
    pool, off, lens = nw.pool_of([s for p in pairs for s in p])
    caps = np.array([nw.nw_cigar_bound(a.size, b.size) for a, b in pairs], np.uint64)
    co = np.concatenate([[0], np.cumsum(caps)]).astype(np.uint64)
    dev = dict(device="cuda")
    s = torch.full((len(pairs),), -1, dtype=torch.int32, **dev)
    e = torch.zeros((len(pairs), 4), dtype=torch.int32, **dev)
    cp = torch.zeros(int(co[-1]), dtype=torch.uint8, **dev)
    cl = torch.zeros(len(pairs), dtype=torch.int64, **dev)
    nw.nw_local_align_batch(ctx, torch.from_numpy(pool).cuda(), off[0::2], lens[0::2], off[1::2], lens[1::2],
                            (1, -1, -1), nw.NW_CIGAR if cigar else 0, s, e, cp if cigar else None,
                            co if cigar else None, cl if cigar else None)

    def read():
        h, n = cp.cpu().numpy(), cl.cpu().numpy()
        text = [bytes(h[int(co[k]):int(co[k]) + int(n[k])]).decode() for k in range(len(pairs))] if cigar else None
        return s.cpu().numpy(), e.cpu().numpy(), text
    return read


@pytest.mark.parametrize("cigar", [True, False])
def test_undone_stripes_are_not_followed(cigar):
    import torch
    import paper_2412_21103_gb300 as nw
    rs = seqgen.Stream(77)

    def family(count, m, n):
        out = []
        for _ in range(count):
            b = rs.bases(max(m, n))
            out.append((seqgen.mutate_distinct(b[:m], rs, 0.08, indel_mean=3.0)[0], b[:n]))
        return out
    with nw.Context(0, torch.cuda.current_stream()) as ctx:
        _call(nw, ctx, family(400, 1500, 9000), cigar)   # late chunks in the slots
        ctx.sync()
        bad = torch.tensor(list(b"ACGTN"), dtype=torch.uint8, device="cuda")
        out = torch.zeros(2, dtype=torch.uint8, device="cuda")
        nw.nw_pack_device(ctx, bad, 5, out)
        _call(nw, ctx, family(400, 1500, 700), cigar)
        with pytest.raises(nw.NWError) as err:
            ctx.sync()
        assert err.value.status == nw.NW_ERR_BAD_BASE
        pairs = family(20, 1100, 900)
        s, e, text = _call(nw, ctx, pairs, cigar)()
        ctx.sync()
        for k, (v, ends, ops) in enumerate(oracle.local_align_many(pairs)):
            assert int(s[k]) == v and tuple(int(x) for x in e[k][2:]) == tuple(ends)[2:], k
            if cigar:
                assert tuple(int(x) for x in e[k]) == tuple(ends) and text[k] == oracle.rle(ops), k
