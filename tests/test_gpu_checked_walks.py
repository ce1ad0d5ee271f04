"""The bounds-checked debug build on the kernels whose stores are checked since
they took over the alignments: the groups of lanes (several passes of a pair,
scorings in units), and the window walk in stretches that join, miss one
another and are walked to their end.  In a fresh process with NW_CHECKS=1;
results are the oracle's and no store is reported out of range."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import os, sys
sys.path.insert(0, ROOT)
import numpy as np, torch
import oracle, seqgen
import paper_2412_21103_gb300 as nw
from paper_2412_21103_gb300 import build
assert nw.lib_path() == build.CHECKS_LIB
build.build(checks=True)
rs = seqgen.Stream(2031)
pairs = []
for k in range(24):
    a = rs.bases(1500 + 61 * k)
    pairs.append((a, seqgen.mutate_distinct(a, rs, 0.08, indel_frac=0.4, indel_mean=3.0)[0]))
    pairs.append((rs.bases(31 * k + 1), rs.bases(700 - 29 * k)))
pool, off, ln = nw.pool_of([s for p in pairs for s in p])
ao, al, bo, bl = off[0::2], ln[0::2], off[1::2], ln[1::2]
os.environ["NW_BAND_KEEP"] = "1"
with nw.Context(0, torch.cuda.current_stream()) as ctx:
    for sc in ((1, -1, -1), (2, -1, -2)):
        want = oracle.align_many(pairs, *sc)
        s, c = nw.nw_align_batch(ctx, pool, ao, al, bo, bl, sc, nw.NW_CIGAR)
        assert s.tolist() == [v for v, _ in want] and c == [oracle.rle(o) for _, o in want], sc
    want = oracle.align_many(pairs)
    for w in (30, 250):
        for stretch in ("1", "2", "7", "72"):
            os.environ["NW_BBAND_STRETCH"] = stretch
            s, c = nw.nw_align_batch_banded(ctx, pool, ao, al, bo, bl, np.full(len(pairs), w, np.uint32), (1, -1, -1),
                                            nw.NW_CIGAR)
            assert s.tolist() == [v for v, _ in want] and c == [oracle.rle(o) for _, o in want], (w, stretch)
    ctx.sync()
print("checked walks ok")
"""


def test_checked_build_of_groups_and_stretched_walks():
    env = dict(os.environ, NW_CHECKS="1")
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CHILD], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0 and "checked walks ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
