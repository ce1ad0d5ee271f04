"""Features of a B whose bit planes come just under the default limit of
shared memory, where the kernel's own words count too: 195,585 to 196,608
bases.  In a fresh process, before any longer B raises the limit for it.  One
4-mer of B matches; a feature is log1p of a whole count over log1p(256), each
within a few units in the last place: 1e-6 absolute."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, ROOT)
import numpy as np, torch
import paper_2412_21103_gb300 as nw
m, n = 5000, int(sys.argv[1])
a, b = np.zeros(m, np.uint8), np.ones(n, np.uint8)
b[100000:100004] = 0
pool, off, lens = nw.pool_of([a, b])
with nw.Context(0, torch.cuda.current_stream()) as ctx:
    f = nw.nw_band_features(ctx, torch.from_numpy(pool).cuda(), off[0:1], lens[0:1], off[1:2], lens[1:2]).cpu().numpy()[0]
W, hist = n // 8, np.zeros(64)
for k in range(256):
    i = (k * (m - 4)) // 255
    c0 = i + int(round((n - m) * i / m))
    if abs(100000 - c0) <= W:
        hist[((100000 - c0 + W) * 64) // (2 * W + 1)] += 1
assert np.allclose(f[:64], np.log1p(hist) / np.log1p(256), rtol=0, atol=1e-6)
print("features ok")
"""


@pytest.mark.parametrize("n", [195584, 195585, 196608, 196609])
def test_features_at_the_default_limit(n):
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CHILD, str(n)], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "features ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
