// Shapes and counts of the bit-sliced score kernel (nw_bits.cu) and of the
// groups of lanes (nw_bits_pair.cu): plain arithmetic, for the host plans and
// the kernels alike.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define NW_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define NW_HOST_DEVICE inline
#endif

namespace nw {

// How a pair of m rows runs: K words a lane, S stripes, and the operations of
// a step.  Chunks in all are counted in 64 bits: two sequences of 2^30 bases
// have 2^23 stripes of 2^25 chunks.
struct BitsShape {
    uint32_t K, S, ops;
    uint32_t period(uint32_t n) const {
        const uint32_t words = (n + 31) / 32;
        return S > 1 && words < K + 3 ? K + 3 : words;
    }
    uint64_t chunks(uint32_t n) const { return (uint64_t)(S - 1) * period(n) + (n + 32 * K + 30) / 32; }
    uint64_t work(uint32_t n) const { return ops * chunks(n); }
};

// The chunk from which on the last stripe's bottom row leaves: its bit 0 is
// column 0 there, and column 32 d - b is bit b of the d-th chunk after it.  Count:
// uint32_t for pairs of fewer than 2^32 chunks, else uint64_t.
template <class Count>
NW_HOST_DEVICE Count bits_last_row(uint32_t S, uint32_t C, uint32_t K) {
    return (Count)(S - 1) * C + K - 1;
}

// The bits [lo, hi] of the d-th chunk from there on that are columns 0 .. n-1 of
// that row (lo > hi: none).  Of chunks before it the difference means nothing.
NW_HOST_DEVICE void bits_last_row_span(uint32_t d, uint32_t n, int32_t &lo, int32_t &hi) {
    const int32_t e = (int32_t)(32u * d), from = (int32_t)(32u * d + 1u - n);
    lo = from > 0 ? from : 0;
    hi = e < 31 ? e : 31;
}

// A pair on G lanes of a warp (a power of two), stripes of 31 rows: its chunks (K in all, from one
// pass of a lane to its next `period`), and its 16-byte record units.  A pair of
// 1.3e14 cells has more than 2^32 chunks; those that a launch takes have records
// that fit the scratch, so their K fits 32 bits.
constexpr uint32_t kPairRows = 31;  // rows per stripe (bits 0..30 of a word)
struct GroupGeom {
    uint32_t S, C, period;
    uint64_t K, rec;
};
inline GroupGeom group_geom(uint32_t m, uint32_t n, uint32_t G) {
    GroupGeom g{};
    if (!m || !n) return g;
    g.S = (m + kPairRows - 1) / kPairRows;
    g.C = (uint32_t)(((uint64_t)n + kPairRows - 1 + 31u) / 32u);
    g.period = g.C > G + 2 ? g.C : G + 2;
    const uint32_t passes = (g.S - 1) >> __builtin_ctz(G);  // (a division, ten times a pair, showed in small batches)
    g.K = (uint64_t)passes * g.period + g.C + ((g.S - 1) & (G - 1));
    g.rec = g.K * 16u * G;
    return g;
}

}  // namespace nw
