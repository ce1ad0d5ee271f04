"""Performance cases: the calls a user of the library makes, at the sizes of its own workloads.

Every case goes through the public entry points of ``paper_2412_21103_gb300`` on one GPU.  A case is a dict of plain
values whose ``"kind"`` names the entry point:

* ``align``    nw_align, one pair on device buffers (score, optionally CIGAR)
* ``batch``    nw_align_batch, many pairs (score-only or CIGAR, device or host buffers, plain or certified learned band)
* ``matrix``   nw_score_all_pairs, all-vs-all scores of a sequence family
* ``star``     nw_center_star, center-star multiple alignment of a family
* ``local``    nw_local_align_batch    * ``affine``  nw_affine_align_batch
* ``serve``    Server: a burst of requests submitted, drained and polled
* ``grad``     nw_band_model_grad, forward and backward of the band network

Sequences are synthetic DNA with the recipes of ``seqgen`` (uniform bases; substitutions, geometric indels and indel
bursts at a divergence drawn per pair), made on the GPU from the seed alone.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2412_21103_gb300 as nw

# Scratch budget of a context: a quarter of the card, so that a program (or a comparison) can hold several.
BUDGET = 64 << 30
LINEAR, GENERAL, AFFINE = (1, -1, -1), (2, -1, -2), (2, -3, -5, -2)


def listed():
    return [
        # The smallest useful call: two unrelated 1,000-base sequences, score and alignment.  Launches and latency count.
        {"name": "align_1k", "kind": "align", "m": 1000, "n": 1000, "related": False, "cigar": True},
        # One long pair: 32,768 bases against a mutated copy (10% substitutions, 2% indels), score and alignment.
        {"name": "align_32k", "kind": "align", "m": 32768, "n": 0, "related": True, "cigar": True},
        # Scoring reads against candidate places: many short pairs, score only.
        {"name": "score_reads", "kind": "batch", "npairs": 20000, "lmin": 50, "lmax": 600, "dmin": 0.01, "dmax": 0.30,
         "general": False, "cigar": False, "learned": False, "host": False},
        # A plain full-grid batch with alignments: genes of 500 to 3,000 bases against their homologues.
        {"name": "batch_cigar", "kind": "batch", "npairs": 3000, "lmin": 500, "lmax": 3000, "dmin": 0.05, "dmax": 0.30,
         "general": False, "cigar": True, "learned": False, "host": False},
        # Another scoring (+2/-1/-2) from and to host memory: a script that hands over numpy arrays and reads strings.
        {"name": "batch_general_host", "kind": "batch", "npairs": 1001, "lmin": 300, "lmax": 2500, "dmin": 0.01,
         "dmax": 0.25, "general": True, "cigar": True, "learned": False, "host": True},
        # The certified learned band: 2,000 to 20,000 bases, 1-25% divergence with indel bursts, score and alignment.
        {"name": "learned_band", "kind": "batch", "npairs": 10000, "lmin": 2000, "lmax": 20000, "dmin": 0.01,
         "dmax": 0.25, "general": False, "cigar": True, "learned": True, "host": False},
        # All-vs-all scores of a 512-sequence family, the launches kept in a CUDA graph (a job that repeats the matrix).
        {"name": "matrix_512", "kind": "matrix", "nseq": 512, "lmin": 500, "lmax": 1500, "graph": True},
        # The multiple alignment of such a family, once: matrix, center, alignments with the center, merged rows.
        {"name": "star_512", "kind": "star", "nseq": 512, "lmin": 500, "lmax": 1500},
        # Finding a mutated window of a reference in a query with flanks: local score, ends and alignment.
        {"name": "local_cigar", "kind": "local", "npairs": 4000, "lmin": 2000, "lmax": 10000, "cigar": True},
        # Affine gaps: 1,000 to 5,000 bases, score and alignment.
        {"name": "affine_cigar", "kind": "affine", "npairs": 2000, "lmin": 1000, "lmax": 5000, "dmin": 0.01,
         "dmax": 0.25, "cigar": True},
        # A burst into the continuous-batching server: lengths 50 to 50,000, half of the requests with an alignment.
        {"name": "serve_burst", "kind": "serve", "npairs": 2000, "lmin": 50, "lmax": 50000, "dmin": 0.01,
         "dmax": 0.30, "workers": 8, "max_batch": 512},
        # One training batch of the band network: gradients and loss.
        {"name": "grad_512", "kind": "grad", "batch": 512},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["align", "batch", "batch", "batch", "matrix", "star", "local", "affine", "serve", "grad"])
    dmin = round(rng.uniform(0.01, 0.15), 3)
    div = {"dmin": dmin, "dmax": round(rng.uniform(dmin, 0.30), 3)}
    if kind == "align":
        return {"kind": kind, "m": _log_int(rng, 64, 32768), "n": 0 if rng.random() < 0.5 else _log_int(rng, 64, 32768),
                "related": True, "cigar": rng.random() < 0.7}
    if kind == "matrix":
        lmin = _log_int(rng, 60, 1000)
        return {"kind": kind, "nseq": _log_int(rng, 8, 512), "lmin": lmin, "lmax": rng.randint(lmin, 1500),
                "graph": rng.random() < 0.5}
    if kind == "star":
        lmin = _log_int(rng, 60, 1000)
        return {"kind": kind, "nseq": _log_int(rng, 8, 512), "lmin": lmin, "lmax": rng.randint(lmin, 1500)}
    if kind == "grad":
        return {"kind": kind, "batch": _log_int(rng, 16, 1024)}
    if kind == "serve":
        lmax = _log_int(rng, 500, 50000)
        return {"kind": kind, "npairs": _log_int(rng, 16, 2000), "lmin": 50, "lmax": lmax, **div,
                "workers": rng.randint(1, 8), "max_batch": _log_int(rng, 32, 1024)}
    if kind == "local":
        lmin = _log_int(rng, 200, 4000)
        return {"kind": kind, "npairs": _log_int(rng, 8, 4000), "lmin": lmin, "lmax": rng.randint(lmin, 10000),
                "cigar": rng.random() < 0.7}
    # pairs: fewer of them where they are long
    lmin = _log_int(rng, 50, 4000 if kind == "batch" else 2500)
    lmax = _log_int(rng, lmin, min(8 * lmin, 20000 if kind == "batch" else 5000))
    most = max(8, min(20000, int(6e9 / (lmax * lmax)) if kind == "affine" else int(1.2e10 / (lmax * lmax))))
    case = {"kind": kind, "npairs": _log_int(rng, 8, most), "lmin": lmin, "lmax": lmax, **div,
            "cigar": rng.random() < 0.6}
    if kind == "batch":
        general = rng.random() < 0.25
        case.update(general=general, learned=not general and lmin >= 1000 and rng.random() < 0.5,
                    host=rng.random() < 0.3)
    return case


# ------------------------------------------------------------------- sequences
class _Seqs:
    """Sequences back to back: codes (uint8, one per base) and lengths (int64), on the GPU."""

    def __init__(self, codes, lens):
        self.codes, self.lens = codes, lens

    def ends(self):
        return torch.cumsum(self.lens, 0)

    def owner(self):
        return torch.repeat_interleave(torch.arange(self.lens.numel(), device=self.lens.device), self.lens)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _rand(g, n):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float32)


def _bases(g, n):
    return torch.randint(0, 4, (int(n),), generator=g, device="cuda", dtype=torch.uint8)


def _log_lens(g, n, lo, hi):
    return torch.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * _rand(g, n)).round().clamp(lo, hi).long()


def _mutate(g, a, rate, indel, bursts):
    """B of every A: events at `rate` (per sequence), a fraction `indel` of them indels (geometric, mean 3), and with
    `bursts` one to three indels of 50 to 500 bases in 30% of the sequences.  Returns B and, per sequence, the score
    of the edits under +1/-1/-1."""
    n, own, ends = a.codes.numel(), a.owner(), a.ends()
    ev, kind = _rand(g, n) < rate[own], _rand(g, n)
    length = 1 + torch.floor(torch.log(1 - _rand(g, n)) / math.log(2.0 / 3.0)).long()
    ins = torch.where(ev & (kind < indel / 2), length, 0)
    start = (ev & (kind >= indel / 2) & (kind < indel)).nonzero().squeeze(1)
    dlen = length[start]
    sub = ev & (kind >= indel)
    if bursts:
        k = a.lens.numel()
        count = torch.where(_rand(g, k) < 0.3, torch.randint(1, 4, (k,), generator=g, device="cuda"), 0)
        who = torch.repeat_interleave(torch.arange(k, device="cuda"), count)
        pos = (ends - a.lens)[who] + (_rand(g, who.numel()) * (a.lens[who] - 1)).long()
        size = torch.randint(50, 501, (who.numel(),), generator=g, device="cuda")
        gone = _rand(g, who.numel()) < 0.5
        ins.index_add_(0, pos, torch.where(gone, 0, size))
        start, dlen = torch.cat([start, pos[gone]]), torch.cat([dlen, size[gone]])
    # deleted ranges end with their sequence, and never take its first base
    first = (ends - a.lens)[own[start]]
    stop = torch.minimum(start + dlen, ends[own[start]])
    start = torch.maximum(start, first + 1)
    ok = stop > start
    cover = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    cover.index_add_(0, start[ok], torch.ones_like(start[ok], dtype=torch.int32))
    cover.index_add_(0, stop[ok], -torch.ones_like(stop[ok], dtype=torch.int32))
    keep = torch.cumsum(cover[:n], 0) == 0
    ins = torch.where(keep, ins, 0)
    sub = sub & keep
    base = torch.where(sub, (a.codes + torch.randint(1, 4, (n,), generator=g, device="cuda", dtype=torch.uint8)) & 3,
                       a.codes)
    per = ins + keep
    place = torch.cumsum(per, 0)
    b = _bases(g, int(place[-1]))
    b[(place - per)[keep]] = base[keep]

    def total(x):
        return torch.zeros(a.lens.numel(), dtype=torch.int64, device="cuda").index_add_(0, own, x.long())

    blen, nsub, nins, nkept = total(per), total(sub), total(ins), total(keep)
    return _Seqs(b, blen), nkept - 2 * nsub - nins - (a.lens - nkept)


def _pairs(seed, count, lmin, lmax, dmin, dmax, bursts, indel=0.2):
    g = _gen(seed)
    lens = _log_lens(g, count, lmin, lmax)
    a = _Seqs(_bases(g, lens.sum()), lens)
    b, score = _mutate(g, a, dmin + (dmax - dmin) * _rand(g, count), indel, bursts)
    return a, b, score


def _family(seed, nseq, lmin, lmax):
    """Mutants of one root's prefixes, 5-30% divergence."""
    g = _gen(seed)
    root = _bases(g, lmax)
    lens = torch.randint(lmin, lmax + 1, (nseq,), generator=g, device="cuda")
    at = torch.arange(int(lens.sum()), device="cuda") - torch.repeat_interleave(torch.cumsum(lens, 0) - lens, lens)
    return _mutate(g, _Seqs(root[at], lens), 0.05 + 0.25 * _rand(g, nseq), 0.2, False)[0]


def _local_pairs(seed, count, lmin, lmax):
    """B random; A a mutated window of B (200 to 2,000 bases, 1-20% divergence) between random flanks of up to 500."""
    g = _gen(seed)
    blen = torch.randint(lmin, lmax + 1, (count,), generator=g, device="cuda")
    b = _Seqs(_bases(g, blen.sum()), blen)
    wmax = torch.clamp(blen, max=2000)
    win = (200 + _rand(g, count) * (wmax - 200)).long().clamp(min=1)
    at = (b.ends() - blen) + (_rand(g, count) * (blen - win)).long()
    inside = torch.arange(int(win.sum()), device="cuda") - torch.repeat_interleave(torch.cumsum(win, 0) - win, win)
    core, _ = _mutate(g, _Seqs(b.codes[torch.repeat_interleave(at, win) + inside], win),
                      0.01 + 0.19 * _rand(g, count), 0.2, False)
    left, right = (torch.randint(0, 501, (count,), generator=g, device="cuda") for _ in range(2))
    alen = left + core.lens + right
    a = _bases(g, alen.sum())
    start = torch.cumsum(alen, 0) - alen + left - (core.ends() - core.lens)
    a[torch.arange(core.codes.numel(), device="cuda") + start[core.owner()]] = core.codes
    return _Seqs(a, alen), b


def _pool(*parts):
    """The packed pool (CUDA uint8; every sequence on a 16-byte boundary) and per part its host offsets and lengths."""
    lens = torch.cat([p.lens for p in parts])
    codes = torch.cat([p.codes for p in parts])
    slot = torch.clamp(((lens + 3) // 4 + 15) // 16 * 16, min=16)
    off = torch.cumsum(slot, 0) - slot
    first = torch.cumsum(lens, 0) - lens
    wide = torch.zeros(int(slot.sum()) * 4, dtype=torch.uint8, device="cuda")
    at = torch.arange(codes.numel(), device="cuda") + torch.repeat_interleave(4 * off - first, lens)
    wide[at] = codes
    q = wide.view(-1, 4)
    pool = q[:, 0] | (q[:, 1] << 2) | (q[:, 2] << 4) | (q[:, 3] << 6)
    hoff, hlen = off.cpu().numpy().astype(np.uint64), lens.cpu().numpy().astype(np.uint32)
    out, k = [], 0
    for p in parts:
        out += [hoff[k:k + p.lens.numel()], hlen[k:k + p.lens.numel()]]
        k += p.lens.numel()
    return (pool.contiguous(), *out)


# ------------------------------------------------------------- the band network
def _labels(a, b, score):
    """log of the smallest half-width whose exit bound lies below the edits' score (+1/-1/-1)."""
    m, n = a.lens.double(), b.lens.double()
    w = (((m + n) / 2 - score.double()) / 1.5 - (n - m).abs()) / 2
    return torch.log(w.clamp(min=8.0)).float()


SHAPES = ((128, 65), (128,), (128, 128), (128,), (128,), (1,))  # W1, b1, W2, b2, W3, b3 of the flat parameters


def _split(p):
    at, out = 0, []
    for shape in SHAPES:
        k = math.prod(shape)
        out.append(p[at:at + k].reshape(shape))
        at += k
    return out


def _initial(seed):
    """Fresh parameters: uniform He weights, zero biases, the output at a half-width of a few hundred."""
    g = _gen(seed)
    flat = torch.zeros(sum(math.prod(x) for x in SHAPES), device="cuda")
    for w, fan in zip(_split(flat)[0::2], (65, 128, 128)):
        w.copy_((torch.rand(w.shape, generator=g, device="cuda") * 2 - 1) * math.sqrt(6.0 / fan))
    flat[-1] = 6.0
    return flat


@functools.lru_cache(maxsize=1)
def _weights():
    """The weights a program keeps: the network trained on 1,024 pairs of a fixed seed."""
    a, b, score = _pairs(9004, 1024, 2000, 20000, 0.01, 0.25, True)
    pool, ao, al, bo, bl = _pool(a, b)
    with nw.Context(0, torch.cuda.current_stream(), BUDGET) as ctx:
        x = nw.nw_band_features(ctx, pool, ao, al, bo, bl)
        ctx.sync()
    t = _labels(a, b, score)
    flat = _initial(9004).requires_grad_(True)
    opt = torch.optim.Adam([flat], lr=2e-3)
    for _ in range(200):
        w1, b1, w2, b2, w3, b3 = _split(flat)
        y = torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ w3 + b3
        opt.zero_grad()
        (0.5 * (y - t).square().mean()).backward()
        opt.step()
    return flat.detach().cpu().numpy()


# ------------------------------------------------------------------ the states
class _State:
    """A context, the inputs and the outputs of one case; a server closes before its context."""

    def __init__(self, case):
        self.case = case
        self.srv = None
        self.ctx = nw.Context(0, torch.cuda.current_stream(), BUDGET)

    def __del__(self):
        if getattr(self, "srv", None) is not None:
            self.srv.close()
        if getattr(self, "ctx", None) is not None:
            self.ctx.close()


def _out(n, dtype=torch.int32):
    return torch.zeros(n, dtype=dtype, device="cuda")


def _cigar_room(al, bl):
    off = np.zeros(len(al) + 1, np.uint64)
    np.cumsum(2 * (al.astype(np.uint64) + bl.astype(np.uint64)) + np.uint64(1), out=off[1:])
    return off


def _cigar_bytes(case):
    """Size of the CIGAR buffer a program allocates once for a kind of call, whatever the sequences of one call: twice
    the bases of both sides, with room for longer pairs and insertions."""
    if case["kind"] == "align":
        return int(2 * (case["m"] + max(case["n"], 1.3 * case["m"] + 64)) + 1)
    if case["kind"] == "star":
        return int(case["nseq"] * (4 * (1.2 * case["lmax"] + 64) + 1))
    count = case["npairs"]
    if case["kind"] == "local":
        return int(count * 2 * (case["lmax"] + 1.3 * 2000 + 1000) + 1)
    per = min(case["lmax"], _mean(case["lmin"], case["lmax"]) * (1 + 8 / math.sqrt(count)))
    return int(count * (4 * 1.25 * per + 3200))


def _case_pairs(case, seed):
    """A, B of a case of pairs."""
    if case["kind"] == "local":
        return _local_pairs(seed, case["npairs"], case["lmin"], case["lmax"])
    if case["kind"] == "align":
        g = _gen(seed)
        a = _Seqs(_bases(g, case["m"]), torch.tensor([case["m"]], device="cuda"))
        if case["related"]:
            b, _ = _mutate(g, a, torch.full((1,), 0.12, device="cuda"), 1.0 / 6.0, False)
            if case["n"]:  # a related sequence of the given length: cut, or longer at its end
                codes = torch.cat([b.codes, _bases(g, case["n"])])[:case["n"]].contiguous()
                b = _Seqs(codes, torch.tensor([case["n"]], device="cuda"))
            return a, b
        return a, _Seqs(_bases(g, case["n"]), torch.tensor([case["n"]], device="cuda"))
    bursts = bool(case.get("learned")) or case["kind"] == "affine"
    return _pairs(seed, case["npairs"], case["lmin"], case["lmax"], case["dmin"], case["dmax"], bursts)[:2]


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind in ("matrix", "star"):
        s.pool, s.off, s.len = _pool(_family(seed, case["nseq"], case["lmin"], case["lmax"]))
        k = case["nseq"]
        if kind == "matrix":
            s.scores = _out((k, k))
            return s
        room = 2 * (s.len.astype(np.uint64) + np.uint64(s.len.max())) + np.uint64(1)
        s.cigar_off = np.concatenate([[0], np.cumsum(room)]).astype(np.uint64)
        s.ld = 8 * case["lmax"] + 64
        s.sums, s.scores = _out(k, torch.int64), _out(k)
        s.cigar = _out(max(_cigar_bytes(case), int(s.cigar_off[-1])), torch.uint8)
        s.cigar_len = _out(k, torch.int64)
        s.msa = _out(k * s.ld, torch.uint8)
        return s
    if kind == "grad":
        a, b, score = _pairs(seed, case["batch"], 2000, 20000, 0.01, 0.25, True)
        pool, ao, al, bo, bl = _pool(a, b)
        nw.nw_band_model_set(s.ctx, _initial(seed).cpu().numpy())
        s.feat, s.target = nw.nw_band_features(s.ctx, pool, ao, al, bo, bl), _labels(a, b, score)
        s.ctx.sync()
        return s
    a, b = _case_pairs(case, seed)
    s.pool, s.ao, s.al, s.bo, s.bl = _pool(a, b)
    if case.get("learned") or kind == "serve":
        nw.nw_band_model_set(s.ctx, _weights())
    if kind == "serve" or case.get("host"):
        s.text = np.zeros(max(_cigar_bytes(case) // 2, 64), np.uint8)
    if kind == "serve":
        s.pool = s.pool.cpu().numpy()
        s.want = np.random.default_rng(seed).random(case["npairs"]) < 0.5
        s.srv = nw.Server(s.ctx, workers=case["workers"], max_batch=case["max_batch"], trace_budget=16 << 30,
                          flags=nw.NW_LEARNED_BAND)
        return s
    if case.get("host"):
        s.pool = s.pool.cpu().numpy()
        return s
    k = len(s.al)
    s.scores = _out(k)
    s.ends = _out((k, 4)) if kind == "local" else None
    s.cigar_off = _cigar_room(s.al, s.bl) if case["cigar"] else None
    s.cigar = _out(max(_cigar_bytes(case), int(s.cigar_off[-1])), torch.uint8) if case["cigar"] else None
    s.cigar_len = _out(k, torch.int64) if case["cigar"] else None
    if kind == "align":
        s.b = s.pool[int(s.bo[0]):]
    return s


def _text(s, cigars):
    """The CIGARs a program reads, back to back in its buffer, and their lengths."""
    text = [c or "" for c in cigars]
    joined = np.frombuffer("".join(text).encode(), np.uint8)
    s.text[:joined.size] = joined
    return s.text, np.array([len(c) for c in text], np.int64)


def run(s):
    case, kind = s.case, s.case["kind"]
    flags = nw.NW_CIGAR if case.get("cigar") else 0
    if kind == "align":
        nw.nw_align(s.ctx, s.pool, int(s.al[0]), s.b, int(s.bl[0]), LINEAR, flags, s.scores, s.cigar, s.cigar_len)
        return [s.scores, s.cigar, s.cigar_len]
    if kind == "batch":
        scoring = GENERAL if case["general"] else LINEAR
        flags |= nw.NW_LEARNED_BAND if case["learned"] else 0
        if case["host"]:
            scores, cigars = nw.nw_align_batch(s.ctx, s.pool, s.ao, s.al, s.bo, s.bl, scoring, flags)
            return [scores, *(_text(s, cigars) if cigars is not None else ())]
        nw.nw_align_batch(s.ctx, s.pool, s.ao, s.al, s.bo, s.bl, scoring, flags, s.scores, s.cigar, s.cigar_off,
                          s.cigar_len)
        return [s.scores, s.cigar, s.cigar_len]
    if kind == "local":
        nw.nw_local_align_batch(s.ctx, s.pool, s.ao, s.al, s.bo, s.bl, LINEAR, flags, s.scores, s.ends, s.cigar,
                                s.cigar_off, s.cigar_len)
        return [s.scores, s.cigar, s.cigar_len, s.ends]
    if kind == "affine":
        nw.nw_affine_align_batch(s.ctx, s.pool, s.ao, s.al, s.bo, s.bl, AFFINE, flags, s.scores, s.cigar, s.cigar_off,
                                 s.cigar_len)
        return [s.scores, s.cigar, s.cigar_len]
    if kind == "matrix":
        return [nw.nw_score_all_pairs(s.ctx, s.pool, s.off, s.len, LINEAR, nw.NW_GRAPH if case["graph"] else 0,
                                      s.scores)]
    if kind == "star":
        center, cols, _ = nw.nw_center_star(s.ctx, s.pool, s.off, s.len, LINEAR, 0, s.sums, s.scores, s.cigar,
                                            s.cigar_off, s.cigar_len, s.msa, s.ld)
        return [s.scores, s.sums, s.cigar, s.cigar_len, s.msa, center, cols]
    if kind == "grad":
        grad, loss = nw.nw_band_model_grad(s.ctx, s.feat, s.target)
        return [grad, loss]
    tickets = s.srv.submit_many(s.pool, s.ao, s.al, s.bo, s.bl, s.want)
    s.srv.drain()
    done = {c[0]: c for c in s.srv.poll_all()}
    done = [done[int(t)] for t in tickets]
    return [np.array([c[2] for c in done], np.int32), *_text(s, [c[3] for c in done]),
            np.array([c[1] for c in done], np.int32)]


# ------------------------------------------------------------------------ work
def _mean_product(lmin, lmax):
    """E[L^2] of a length log-uniform in [lmin, lmax]."""
    r = math.log(lmax / lmin)
    return (lmax ** 2 - lmin ** 2) / (2 * r) if r > 1e-9 else float(lmax) ** 2


def _mean(lmin, lmax):
    r = math.log(lmax / lmin)
    return (lmax - lmin) / r if r > 1e-9 else float(lmax)


def work(case):
    """Bytes: packed sequences in, scores and alignments out.  Operations: the textbook cell's four (select, diagonal
    add, larger gap move, add-max; six with affine gaps) on every cell of the grid; for the certified band on the
    cells of the narrowest band that certifies (half-width about 0.8 of the divergence times the length)."""
    kind = case["kind"]
    if kind == "grad":
        n = case["batch"]
        p = sum(math.prod(x) for x in SHAPES)
        return {"bytes": 4 * (n * 66 + 2 * p + 1), "flops": 6 * n * p}
    if kind in ("matrix", "star"):
        k, length = case["nseq"], (case["lmin"] + case["lmax"]) / 2
        cells = k * (k - 1) / 2 * length * length
        if kind == "matrix":
            return {"bytes": k * length / 4 + 4 * k * k, "flops": 4 * cells}
        return {"bytes": k * length / 4 + k * (2 * length + 20), "flops": 4 * (cells + k * length * length)}
    if kind == "align":
        m, n, count = case["m"], case["n"] or case["m"], 1
        cells, bases = float(m) * n, float(m + n)
    elif kind == "local":
        count, n = case["npairs"], (case["lmin"] + case["lmax"]) / 2
        m = 500 + (200 + min(n, 2000)) / 2
        cells, bases = count * m * n, count * (m + n)
    else:
        count = case["npairs"]
        cells = count * _mean_product(case["lmin"], case["lmax"])
        bases = 2 * count * _mean(case["lmin"], case["lmax"])
        if case.get("learned") or kind == "serve":
            cells *= min(1.0, 1.6 * (case["dmin"] + case["dmax"]) / 2)
    share = 0.5 if kind == "serve" else 1.0 if case["cigar"] else 0.0
    return {"bytes": bases / 4 + 4 * count + share * (0.4 * bases + 8 * count),
            "flops": (6 if kind == "affine" else 4) * cells}


# ------------------------------------------------------- the results in 64 bits
def _scores64(a, b, match, mismatch, gap):
    """Global alignment scores by anti-diagonals over int64 grids, all pairs at once."""
    k, lm, ln = a.lens.numel(), int(a.lens.max()), int(b.lens.max())

    def padded(s, width, fill):
        out = torch.full((k, width), fill, dtype=torch.int64, device="cuda")
        at = torch.arange(s.codes.numel(), device="cuda") - torch.repeat_interleave(s.ends() - s.lens, s.lens)
        out[s.owner(), at] = s.codes.long()
        return out

    av, bv = padded(a, lm, 4), padded(b, ln, 5).flip(1)
    far = -(1 << 40)
    rows = torch.arange(lm + 1, device="cuda")
    prev2 = torch.full((k, lm + 1), far, dtype=torch.int64, device="cuda")
    prev = prev2.clone()
    prev[:, 0] = 0
    out = torch.where((a.lens + b.lens) == 0, 0, torch.full_like(a.lens, far))
    for d in range(1, lm + ln + 1):
        cur = torch.full_like(prev, far)
        cur[:, 1:] = prev[:, :-1] + gap
        cur = torch.maximum(cur, prev + gap)
        lo, hi = max(1, d - ln), min(lm, d - 1)
        if lo <= hi:
            same = av[:, lo - 1:hi] == bv[:, ln - d + lo:ln - d + hi + 1]
            cur[:, lo:hi + 1] = torch.maximum(cur[:, lo:hi + 1],
                                              prev2[:, lo - 1:hi] + torch.where(same, match, mismatch))
        cur[:, (rows > d) | (rows < d - ln)] = far
        here = (a.lens + b.lens) == d
        out = torch.where(here, cur.gather(1, a.lens.unsqueeze(1)).squeeze(1), out)
        prev2, prev = prev, cur
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "grad":
        s = prepare(case, seed)
        x, t = s.feat.to(torch.bfloat16).double(), s.target.double()

        def rounded(v):  # the network's activations are BF16; the rounding passes gradients through
            return v + (v.detach().float().to(torch.bfloat16).double() - v.detach())

        flat = _initial(seed).double().requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = _split(flat)
        w1, w2, w3 = rounded(w1), rounded(w2), rounded(w3)
        h1 = rounded(torch.relu(x @ w1.T + b1))
        h2 = rounded(torch.relu(h1 @ w2.T + b2))
        loss = 0.5 * (h2 @ w3 + b3 - t).square().mean()
        loss.backward()
        return [flat.grad, loss.detach().reshape(1)]
    if kind not in ("align", "batch"):
        return None
    # scores of the smaller cases; alignments are bytes
    a, b = _case_pairs(case, seed)
    steps = int(a.lens.max() + b.lens.max())
    if steps > 8000 or steps * a.lens.numel() * int(a.lens.max()) > 2e10:
        return None
    scores = _scores64(a, b, *(GENERAL if case.get("general") else LINEAR))
    return [scores, *([None, None] if case["cigar"] else [])]
