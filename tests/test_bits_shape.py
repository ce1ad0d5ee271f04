"""Shapes and column counts of the bit-sliced score kernel and of the groups of
lanes (nw_bits_shape.h), compiled for the host, against Python's integers:
where the columns of the last stripe's bottom row leave, for sizes up to the
accepted 2^30 bases, that the chunks of a pair hand out each of its columns
exactly once, and the chunks and records of a pair on a group."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_21103_gb300", "csrc")
SOURCE = r"""
#include "nw_bits_shape.h"
template <class Count>
void span_of(Count c, uint32_t S, uint32_t C, uint32_t K, uint32_t n, int32_t *out) {
    const Count last = nw::bits_last_row<Count>(S, C, K);
    nw::bits_last_row_span((uint32_t)(c - last), n, out[0], out[1]);
    if (c < last) out[0] = 1, out[1] = 0;
}
extern "C" {
void span(uint64_t c, uint32_t S, uint32_t C, uint32_t K, uint32_t n, int32_t *out) { span_of<uint64_t>(c, S, C, K, n, out); }
void span32(uint32_t c, uint32_t S, uint32_t C, uint32_t K, uint32_t n, int32_t *out) { span_of<uint32_t>(c, S, C, K, n, out); }
uint32_t period(uint32_t K, uint32_t S, uint32_t n) { return nw::BitsShape{K, S, 10 * K + 6}.period(n); }
uint64_t chunks(uint32_t K, uint32_t S, uint32_t n) { return nw::BitsShape{K, S, 10 * K + 6}.chunks(n); }
uint64_t group(uint32_t m, uint32_t n, uint32_t G, uint64_t *rec) {
    const nw::GroupGeom g = nw::group_geom(m, n, G);
    *rec = g.rec;
    return g.K;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("shape")
    (d / "shape.cpp").write_text(SOURCE)
    so = str(d / "shape.so")
    cxx = shutil.which("g++") or shutil.which("c++")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(d / "shape.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.span.argtypes = [ctypes.c_uint64] + [ctypes.c_uint32] * 4 + [ctypes.POINTER(ctypes.c_int32)]
    lib.span32.argtypes = [ctypes.c_uint32] * 5 + [ctypes.POINTER(ctypes.c_int32)]
    lib.period.restype, lib.chunks.restype, lib.group.restype = ctypes.c_uint32, ctypes.c_uint64, ctypes.c_uint64
    return lib


def _span(lib, c, S, C, K, n):
    out, out32 = (ctypes.c_int32 * 2)(), (ctypes.c_int32 * 2)()
    lib.span(c, S, C, K, n, out)
    if lib.chunks(K, S, n) < 1 << 32:  # the form the kernel takes then
        lib.span32(c, S, C, K, n, out32)
        assert (out32[0], out32[1]) == (out[0], out[1]) or (out32[0] > out32[1] and out[0] > out[1])
    return out[0], out[1]


def _want(c, S, C, K, n):
    e = 32 * (c - (S - 1) * C - K + 1)
    lo, hi = max(e + 1 - n, 0), min(31, e)
    return (lo, hi) if lo <= hi else None


SIZES = [(m, n) for m in (1, 130, 5000, 750_000, 4_200_000, (1 << 30) - 1) for n in (1, 33, 700, 750_001, (1 << 30) - 1)]


@pytest.mark.parametrize("K", [1, 2, 4])
def test_columns_of_large_pairs(lib, K):
    for m, n in SIZES:
        S = -(-m // (32 * K))
        C = max(-(-n // 32), K + 3) if S > 1 else -(-n // 32)
        T = (S - 1) * C + (n + 32 * K + 30) // 32
        assert lib.period(K, S, n) == C and lib.chunks(K, S, n) == T
        first, some = (S - 1) * C + K - 1, set(range(min(T, 40)))
        some |= {c + d for c in (first, T - 1) for d in range(-3, 4)}
        # chunks whose 32 c differs from the last stripe's by a multiple of 2^32
        some |= {first - k * (1 << 27) + d for k in (1, 2, 5) for d in (0, 1, C // 2, C)}
        for c in some:
            if 0 <= c < T:
                lo, hi = _span(lib, c, S, C, K, n)
                assert ((lo, hi) if lo <= hi else None) == _want(c, S, C, K, n), (m, n, c)


@pytest.mark.parametrize("K", [1, 2, 4])
def test_every_column_once(lib, K):
    for S in (1, 2, 5):
        for n in (1, 31, 32, 33, 63, 64, 65, 97, 500):
            C, T = lib.period(K, S, n), lib.chunks(K, S, n)
            cols = []
            for c in range(T):
                lo, hi = _span(lib, c, S, C, K, n)
                cols += [32 * (c - (S - 1) * C - K + 1) - b for b in range(lo, hi + 1)]
            assert sorted(cols) == list(range(n)), (S, n)


def test_chunks_and_records_of_a_group(lib):
    # the last pair: 127 passes of 2^25 chunks and one more, 2^32 in all
    for m, n in SIZES + [(0, 5), (5, 0), (31, 1), (32, 2), (993, 1025), (31 * 4064 + 1, (1 << 30) - 61)]:
        for G in (1, 4, 32):
            S, C = -(-m // 31), (n + 61) // 32
            K = (S - 1) // G * max(C, G + 2) + C + (S - 1) % G if m and n else 0
            rec = ctypes.c_uint64()
            assert lib.group(m, n, G, ctypes.byref(rec)) == K and rec.value == K * 16 * G, (m, n, G)
