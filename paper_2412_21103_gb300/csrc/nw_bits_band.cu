// Bit-sliced certified band (a8) with pointers (a4) and its walk (a5).
//
// The fill is the difference form of nw_bits.cu (dH, dV in two bit planes,
// T = max(s', a, b), dV = T - a, dH = T - b) on a window that follows the
// band: on anti-diagonal a the window holds the Hw = 32*g*Q rows
// r0(a) .. r0(a)+Hw-1 with r0(a) = floor((a - hi)/2), so it moves down one
// row every second anti-diagonal and always covers the band's diagonals
// [lo, hi] (2*Hw >= hi - lo + 4).  A pair belongs to a group of g lanes
// (1..32, a power of two) holding Q words each, the lane's 32*Q rows dealt
// out to them in turn: bit p of word v of lane l is window row P = 32*Q*l +
// Q*p + v, which is row r0(a) + P, column a - r0(a) - P.
//
// Anti-diagonals come in pairs: a step where r0 stays (the B bases slide one
// row down, a new column enters at the top; the cell above is row P - 1 of the
// previous anti-diagonal, the cell to its left the same row) and a step where
// r0 grows (the A bases slide one row up, a new row enters at the bottom; the
// cell above is the same row, the cell to the left row P + 1).  A row's
// neighbours are the same bit of the neighbouring words, so of a lane's Q words
// one is shifted (the first by the last one's upper, the last by the first
// one's lower neighbours) and the bases change their words' roles; across
// lanes of a group through warp shuffles.  Cells just outside the window
// take the values of a gap move from a computed neighbour, which a real
// path reaches: above the top row a horizontal extension (dH = 0), below
// the bottom row a vertical one (dV = 0).  Every computed value is therefore
// reached by some path (never above the full grid's value) and at least the
// value of the DP restricted to the window, which contains the band -- so the
// certificate of the scalar banded kernels holds unchanged: a score above
// the exit bound U0 of the band equals the full score, and the walk below
// gives the full grid's alignment.  Cells of row 0 or column 0 and beyond
// (the grid's boundary) get s' = 0 through a mask in the ramp chunks, which
// keeps their differences at 0.
//
// The score is tracked at the window's bottom cell (its dH on a step without a
// shift, its dV on a shift) and carried up the last anti-diagonal to (m, n).
//
// Alignments.  The fill writes no pointers: every block of kBlockChunks chunks
// (64 anti-diagonals) it keeps the window's four planes (16 bytes per word).
// The walk then goes back block by block: it recomputes the pointer bits of the
// block it stands in from the planes kept at its start -- only the 128 rows
// around the path, because a cell of an anti-diagonal depends on the row
// itself and its two neighbours one anti-diagonal pair earlier, so nothing
// further than 32 rows away reaches the path within a block -- into shared
// memory and follows the path through them.  Long paths are walked in
// stretches side by side, from guessed cells whose paths soon run into the
// one looked for (see BitsWalker).  Pointer bits, per cell:
// L = T != s' (the diagonal loses), and Hb = dV != 0 (the vertical move
// loses); the walk reads !L -> diagonal, else !Hb -> vertical, else
// horizontal, the diagonal > vertical > horizontal order of the scalar
// kernels.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <type_traits>
#include <vector>

#include "nw_bits.cuh"
#include "nw_order.h"

namespace nw {

// Words per lane: at most 4, so a pair's window holds up to 128 words (4,096
// rows, bands up to ~8,190 diagonals).  Up to 8 words per lane (fewer lanes
// per pair, the lane's fixed work per step shared by more words) measured 1.5x
// slower on the band workload while every word shifted; with dealt rows the
// lane's share is 14 of 94 instructions, and the longest pair's time counts.
constexpr int kBandBitsMaxQ = 4;
constexpr int kBandBitsMaxWords = 32 * kBandBitsMaxQ;
// Anti-diagonals between kept planes: kBlockChunks chunks of 64; the walk's
// sub-window of kSubWords words covers the rows a block's path can depend on
// (kBlockSteps on either side of it), wherever in a word the path stands.
constexpr int kBlockChunks = 1;
constexpr int kSubWords = 4;
constexpr int kSubPairs = 32 / kSubWords;                // pairs per warp of the walk
constexpr int kBlockSteps = 32 * kBlockChunks;           // pairs of anti-diagonals per block
static_assert(kSubWords * 32 >= 2 * kBlockSteps + 1 + 31 + 16, "the sub-window must hold a block's dependencies");
// Records of a pair's block in shared memory, 16 bytes each; the padding sets
// neighbouring groups' records on different banks.
constexpr int kTileRecs = kBlockSteps * kSubWords + 4;
// Diagonal moves a lane looks ahead in one pass of the walk.
constexpr int kAhead = 16 / kSubWords;
// Blocks of a stretch of a walk (see BitsWalker).  Walks of both rounds, pairs of
// 2-20 kb, stretches of 25 / 50 / 75 / 100 / 150 blocks: 10,000 pairs 5.3 / 3.8 /
// 3.6 / 4.0 / 4.3 ms (whole pairs: 8.0), 2,500 pairs 2.9 / 2.3 / 2.4 / 3.0 / 3.2.
constexpr uint32_t kStretch = 72;
// Warps per CTA of the fill: one per scheduler.
constexpr int kBandWarps = 4;

struct BandBitsTask {
    int64_t a_slot, b_slot; // planar slots of A (rows) and B (columns)
    uint64_t ptr_off;       // first kept planes of the pair (16-byte units)
    uint32_t m, n;
    int32_t hi;             // window anchor: the band's upper diagonal, raised to the parity of m+n
    int32_t a_first;        // first anti-diagonal (a step without a shift), <= 0
    uint32_t nchunks;       // chunks of 64 anti-diagonals; the last ends at m+n
    uint32_t out0;          // the caller's score slot
};

struct BandBitsJob {
    uint32_t t0, cnt;  // tasks [t0, t0 + cnt), one per group of g lanes
    uint32_t g, Q;     // lanes per pair, words per lane
    uint32_t nchunks;  // the job's largest
};

struct BandBitsArgs {
    const uint32_t *pl0, *pl1;
    int64_t max_base;  // largest global base index a window load may start at
    const BandBitsTask *tasks;
    const BandBitsJob *jobs;
    uint32_t njobs;
    uint32_t *counter;
    uint4 *ptr;         // kept planes (H0, H1, V0, V1), per pair [block][word]
    uint64_t ptr_cap;   // 16-byte units at ptr (checked build)
    int32_t *scores;
    int32_t *gathered;  // per task, in task order
    uint32_t score_cap;
    int32_t gap;
    uint32_t two, half;  // 2 and 2^31: as arguments, so that products by them stay multiplies
    uint32_t *err;
};

// Bits b of a word with lo <= b <= hi (empty when hi < lo); PTX shifts
// clamp at the register width.
__device__ __forceinline__ uint32_t range_mask(int32_t lo, int32_t hi) {
    uint32_t a, b;
    asm("shl.b32 %0, %1, %2;" : "=r"(a) : "r"(~0u), "r"((uint32_t)max(lo, 0)));
    asm("shl.b32 %0, %1, %2;" : "=r"(b) : "r"(~0u), "r"((uint32_t)max(hi + 1, 0)));
    return a & ~b;
}

// The cells of one word: inputs a (dH above), b (dV to the left), bases A,
// B, mask mk of cells inside the grid (all ones unless RAMP; the others keep
// the boundary's zero differences); outputs the new planes and, with PTR, the
// pointer bits.  The paper's scoring: s' = 3 (match) or 1, where T != s'
// exactly where the bases differ and a or b is 2 or 3.
template <bool RAMP, bool PTR>
__device__ __forceinline__ void band_cell(uint32_t A0, uint32_t A1, uint32_t B0, uint32_t B1, uint32_t a0,
                                          uint32_t a1, uint32_t b0, uint32_t b1, uint32_t mk, uint32_t &H0,
                                          uint32_t &H1, uint32_t &V0, uint32_t &V1, uint32_t &L, uint32_t &Hb) {
    const uint32_t eq = lop3<kLutEq>(A0, B0, A1 ^ B1);
    if constexpr (PTR) L = lop3<kLutOrAndNot>(a1, b1, eq);
    bits_cell(eq, a0, a1, b0, b1, H0, H1, V0, V1);
    if constexpr (RAMP) {
        H0 &= mk;
        H1 &= mk;
        V0 &= mk;
        V1 &= mk;
    }
    if constexpr (PTR) Hb = V0 | V1;
}

// Masks of a lane's rows lo .. hi (counted from its first) by word.
template <int Q>
struct RowMask {
    int32_t ql, rl, qh, rh;
    __device__ RowMask(int32_t lo, int32_t hi) {
        lo = max(lo, -1);
        hi = max(hi, -1);
        ql = (int32_t)((uint32_t)(lo + Q) / Q) - 1;
        rl = lo - Q * ql;
        qh = (int32_t)((uint32_t)(hi + Q) / Q) - 1;
        rh = hi - Q * qh;
    }
    __device__ uint32_t operator()(int v) const { return range_mask(ql + (v < rl), qh - (v > rh)); }
};

// A lane's Q words of the window: difference planes and bases, and the bases
// that enter it during a chunk: the next columns above its rows (inB, the
// first at bit 31) and the next rows below (inA, the first at bit 0).  The
// bases stay in place while rows slide over them: after k steps row v of the
// A side is word (v + k) mod Q, of the B side word (v - k) mod Q, and a step
// moves one word of each by one bit.
template <int Q>
struct BandWords {
    uint32_t A0[Q], A1[Q], B0[Q], B1[Q], H0[Q], H1[Q], V0[Q], V1[Q];
    uint32_t inA0, inA1, inB0, inB1;
};

// The planar bases as the window reads them (clamped: bases outside belong to no cell that matters).
struct BandBases {
    const uint32_t *pl0, *pl1;
    int64_t max_base, Ag, Bg;
    __device__ uint32_t at(const uint32_t *pl, int64_t g) const {
        return plane_window(pl, min(max(g, -kPlanePad), max_base));
    }
    // words of 32 rows from row r on, and of 32 columns from column c down (bit 0 = the first)
    __device__ uint2 rows(int32_t r) const {
        const int64_t g = Ag + r - 1;
        return make_uint2(at(pl0, g), at(pl1, g));
    }
    __device__ uint2 cols(int32_t c) const {
        const int64_t g = Bg + c - 32;
        return make_uint2(__brev(at(pl0, g)), __brev(at(pl1, g)));
    }
};

// x * k + c, the high word.
__device__ __forceinline__ uint32_t muladd_hi(uint32_t x, uint32_t k, uint32_t c) {
    uint32_t d;
    asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(x), "r"(k), "r"(c));
    return d;
}

// A pair of anti-diagonals, the k-th (mod Q) of its chunk, of a window spread
// over groups of g lanes.  The first has the lane's first row at row r and
// columns 1 .. at rows below cmax; nzt, nzb: 0 on the group's top / bottom
// lane, else 1; half: 2^31.  bottom() runs after the first with the lane's last
// H word, after the second with its last V word (the score's path); rec(v, L,
// Hb, L', Hb') takes the pointer bits.
//
// What bounds it: the logic pipe, 10 operations per word and anti-diagonal
// (12 with pointers) and 4 per lane; the choice at the group's ends and the
// entering bases' shifts are multiplies, which issue beside it.  At one warp
// per scheduler the fill keeps it 70% busy.  10,000 pairs of 2-20 kb, both
// rounds: 10.3 ms, with words of 32 consecutive rows and 14 operations 11.5.
template <int Q, int k, bool RAMP, bool PTR, class Bottom, class Rec>
__device__ __forceinline__ void band_two(BandWords<Q> &w, uint32_t g, uint32_t nzt, uint32_t nzb, uint32_t half,
                                         int32_t r, int32_t cmax, Bottom bottom, Rec rec) {
    constexpr auto mod = [](int x) { return ((x % Q) + Q) % Q; };
    uint32_t Ln[Q], Hn[Q];
    {
        // no shift; above the window a horizontal gap, dH = 0
        const uint32_t sH0 = mul(__shfl_up_sync(kFull, w.H0[Q - 1], 1, g), nzt);
        const uint32_t sH1 = mul(__shfl_up_sync(kFull, w.H1[Q - 1], 1, g), nzt);
        constexpr int nb = mod(-(k + 1));  // the new first row's bases
        w.B0[nb] = __funnelshift_l(w.inB0, w.B0[nb], 1);
        w.B1[nb] = __funnelshift_l(w.inB1, w.B1[nb], 1);
        w.inB0 = mul(w.inB0, 2u);
        w.inB1 = mul(w.inB1, 2u);
        const uint32_t f0 = __funnelshift_l(sH0, w.H0[Q - 1], 1), f1 = __funnelshift_l(sH1, w.H1[Q - 1], 1);
        const RowMask<Q> mk(RAMP ? 1 - r : 0, RAMP ? cmax - 1 : 0);
#pragma unroll
        for (int v = Q - 1; v >= 0; --v) {
            const int vb = mod(v - (k + 1)), va = mod(v + k);
            const uint32_t a0 = v ? w.H0[v ? v - 1 : 0] : f0, a1 = v ? w.H1[v ? v - 1 : 0] : f1;
            band_cell<RAMP, PTR>(w.A0[va], w.A1[va], w.B0[vb], w.B1[vb], a0, a1, w.V0[v], w.V1[v],
                                 RAMP ? mk(v) : ~0u, w.H0[v], w.H1[v], w.V0[v], w.V1[v], Ln[v], Hn[v]);
        }
        bottom(w.H0[Q - 1], w.H1[Q - 1]);
    }
    {
        // shift; below the window a vertical gap, dV = 0
        const uint32_t sV0 = mul(__shfl_down_sync(kFull, w.V0[0], 1, g), nzb);
        const uint32_t sV1 = mul(__shfl_down_sync(kFull, w.V1[0], 1, g), nzb);
        constexpr int na = mod(k);  // the new last row's bases
        w.A0[na] = __funnelshift_r(w.A0[na], w.inA0, 1);
        w.A1[na] = __funnelshift_r(w.A1[na], w.inA1, 1);
        w.inA0 = muladd_hi(w.inA0, half, 0u);
        w.inA1 = muladd_hi(w.inA1, half, 0u);
        const uint32_t f0 = __funnelshift_r(w.V0[0], sV0, 1), f1 = __funnelshift_r(w.V1[0], sV1, 1);
        const RowMask<Q> mk(RAMP ? -r : 0, RAMP ? cmax - 1 : 0);
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            const int vb = mod(v - (k + 1)), va = mod(v + k + 1);
            const uint32_t b0 = v + 1 < Q ? w.V0[v + 1 < Q ? v + 1 : 0] : f0;
            const uint32_t b1 = v + 1 < Q ? w.V1[v + 1 < Q ? v + 1 : 0] : f1;
            uint32_t Ls = 0, Hs = 0;
            band_cell<RAMP, PTR>(w.A0[va], w.A1[va], w.B0[vb], w.B1[vb], w.H0[v], w.H1[v], b0, b1,
                                 RAMP ? mk(v) : ~0u, w.H0[v], w.H1[v], w.V0[v], w.V1[v], Ls, Hs);
            if constexpr (PTR) rec(v, Ln[v], Hn[v], Ls, Hs);
        }
        bottom(w.V0[Q - 1], w.V1[Q - 1]);
    }
}

// The 32 pairs of a chunk; step(d, k) runs pair d = k mod Q.
template <int Q, class Step>
__device__ __forceinline__ void band_chunk(BandWords<Q> &w, Step step) {
    constexpr int U = Q == 3 ? 3 : 4;  // pairs per turn of the loop: the words' roles come round
    int d = 0;
#pragma unroll 1
    for (; d + U <= 32; d += U) {
        step(d, std::integral_constant<int, 0>{});
        step(d + 1, std::integral_constant<int, 1 % Q>{});
        step(d + 2, std::integral_constant<int, 2 % Q>{});
        if constexpr (U == 4) step(d + 3, std::integral_constant<int, 3 % Q>{});
    }
    if constexpr (Q == 3) {
        step(30, std::integral_constant<int, 0>{});
        step(31, std::integral_constant<int, 1>{});
        // 32 pairs on: row v of A is word v + 2, of B word v - 2
        const uint32_t a0[3] = {w.A0[2], w.A0[0], w.A0[1]}, a1[3] = {w.A1[2], w.A1[0], w.A1[1]};
        const uint32_t b0[3] = {w.B0[1], w.B0[2], w.B0[0]}, b1[3] = {w.B1[1], w.B1[2], w.B1[0]};
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            w.A0[v] = a0[v];
            w.A1[v] = a1[v];
            w.B0[v] = b0[v];
            w.B1[v] = b1[v];
        }
    }
}

// Every Q-th bit of Q words of consecutive rows, from bit v on (they go to word v).
template <int Q>
__device__ __forceinline__ uint32_t deal_word(const uint32_t (&c)[Q], int v) {
    uint32_t out = 0;
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        const int x0 = (v + 32 * (Q - j)) % Q;  // the first of the word's rows that goes to word v
        int p = (32 * j + x0) / Q;
#pragma unroll 1
        for (int x = x0; x < 32; x += Q, ++p) out |= ((c[j] >> x) & 1u) << p;
    }
    return out;
}

// The way back: the 32 rows from row 32*j of a lane's rows on, from its Q words
// of one plane.
__device__ __forceinline__ uint32_t collect_rows(const uint32_t (&w)[kBandBitsMaxQ], uint32_t Q, uint32_t j) {
    if (Q == 1) return w[0];
    uint32_t out = 0;
    if (Q == 2) {
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            uint32_t x = (w[v] >> (16 * j)) & 0xFFFFu;
            x = (x | x << 8) & 0x00FF00FFu;
            x = (x | x << 4) & 0x0F0F0F0Fu;
            x = (x | x << 2) & 0x33333333u;
            x = (x | x << 1) & 0x55555555u;
            out |= x << v;
        }
    } else if (Q == 4) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            uint32_t x = (w[v] >> (8 * j)) & 0xFFu;
            x = (x | x << 12) & 0x000F000Fu;
            x = (x | x << 6) & 0x03030303u;
            x = (x | x << 3) & 0x11111111u;
            out |= x << v;
        }
    } else {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const uint32_t o = ((uint32_t)v + 3u - (32u * j) % 3u) % 3u;  // the first of the rows in word v
            uint32_t x = (w[v] >> ((32u * j + o) / 3u)) & 0x7FFu;
            x = (x | x << 16) & 0x070000FFu;
            x = (x | x << 8) & 0x0700F00Fu;
            x = (x | x << 4) & 0x430C30C3u;
            x = (x | x << 2) & 0x49249249u;
            out |= x << o;
        }
    }
    return out;
}

template <int Q, bool KEEP>
__device__ __forceinline__ void band_job(const BandBitsArgs &p, const BandBitsJob &job, uint32_t lane) {
    const uint32_t g = job.g;
    const uint32_t gl = lane & (g - 1), grp = lane / g;
    const bool active = grp < job.cnt;
    const uint32_t tid = job.t0 + (active ? grp : 0u);
    const BandBitsTask t = p.tasks[tid];
    const int32_t gq = (int32_t)g * Q, Hw = 32 * gq, wo = 32 * (int32_t)gl * Q;  // wo: the lane's first row in the window
    const int32_t a0 = t.a_first;
    const int32_t R = (a0 - t.hi - 1) >> 1;  // r0(a_first); a_first - hi is odd
    const BandBases bs{p.pl0, p.pl1, p.max_base, t.a_slot, t.b_slot};
    BandWords<Q> w;
    {
        uint32_t a[2][Q], b[2][Q];
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            const uint2 x = bs.rows(R + wo + 32 * v), y = bs.cols(a0 - 1 - R - wo - 32 * v);
            a[0][v] = x.x;
            a[1][v] = x.y;
            b[0][v] = y.x;
            b[1][v] = y.y;
        }
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            w.A0[v] = deal_word<Q>(a[0], v);
            w.A1[v] = deal_word<Q>(a[1], v);
            w.B0[v] = deal_word<Q>(b[0], v);
            w.B1[v] = deal_word<Q>(b[1], v);
            w.H0[v] = w.H1[v] = w.V0[v] = w.V1[v] = 0;
        }
    }
    // the bases that enter the lane's rows during a chunk, loaded one chunk ahead
    uint2 fa = bs.rows(R + wo + 32 * Q), fb = bs.cols(a0 - R - wo + 31);
    const uint32_t nzt = gl == 0 ? 0u : 1u, nzb = gl == g - 1 ? 0u : 1u;  // 0 on the group's top / bottom lane
    uint32_t low0 = 0, low1 = 0;  // W of the window's bottom cell: low0 + 2 * low1
    const uint32_t nch = t.nchunks;
    const uint32_t gmask = g == 32 ? kFull : (((1u << g) - 1u) << (grp * g));
    uint4 *kp = KEEP ? p.ptr + t.ptr_off + gl * Q : nullptr;  // this lane's kept planes of the next block
    uint32_t keep_in = 0;                                     // chunks until the next block starts
    for (uint32_t c = 0; c < job.nchunks; ++c) {
        const bool live = active && c < nch;
        const int32_t rc = R + 32 * (int32_t)c, ac = a0 + 64 * (int32_t)c;  // r0 and a of the chunk's first step
        if constexpr (KEEP) {
            if (keep_in == 0) {
                keep_in = kBlockChunks;
#pragma unroll
                for (int v = 0; v < Q; ++v)
                    if (live && in_range((uint64_t)(kp - p.ptr) + v, p.ptr_cap, p.err, kSiteBandBitsPtr))
                        __stcg(kp + v, make_uint4(w.H0[v], w.H1[v], w.V0[v], w.V1[v]));
                kp += gq;
            }
            --keep_in;
        }
        w.inA0 = fa.x;
        w.inA1 = fa.y;
        w.inB0 = fb.x;
        w.inB1 = fb.y;
        fa = bs.rows(rc + 32 + wo + 32 * Q);
        fb = bs.cols(ac + 64 - (rc + 32) - wo + 31);
        // masks only while some cell of the chunk lies on or beyond row 0 / column 0
        const bool ramp = __any_sync(kFull, live && !(rc >= 1 && ac - rc - Hw >= 0));
        auto steps = [&](auto ramp_tag) {
            band_chunk<Q>(w, [&](int d, auto k) {
                band_two<Q, decltype(k)::value, decltype(ramp_tag)::value, false>(
                    w, g, nzt, nzb, p.half, rc + d + wo, ac - rc + d - wo,
                    [&](uint32_t x0, uint32_t x1) {
                        low0 = muladd_hi(x0, p.two, low0);
                        low1 = muladd_hi(x1, p.two, low1);
                    },
                    [](int, uint32_t, uint32_t, uint32_t, uint32_t) {});
            });
        };
        if (ramp) steps(std::true_type{});
        else steps(std::false_type{});
        if (active && c + 1 == nch) {
            // W(m, n): the bottom cell, then up the last anti-diagonal: each row
            // takes off its cell's dV and adds the dH of the cell above it
            const int32_t Pm = (int32_t)t.m - (R + 32 * (int32_t)nch);
            int32_t sum = gl == g - 1 ? (int32_t)(low0 + 2 * low1) : 0;
            const RowMask<Q> vm(Pm + 1 - wo, Hw - 1 - wo), hm(Pm - wo, Hw - 2 - wo);
#pragma unroll
            for (int v = 0; v < Q; ++v)
                sum += __popc(w.H0[v] & hm(v)) + 2 * __popc(w.H1[v] & hm(v)) - __popc(w.V0[v] & vm(v)) -
                       2 * __popc(w.V1[v] & vm(v));
            for (uint32_t o = 1; o < g; o <<= 1) sum += __shfl_xor_sync(gmask, sum, o);
            if (gl == 0) {
                const int32_t sc = sum + p.gap * (int32_t)(t.m + t.n);
                if (in_range(t.out0, p.score_cap, p.err, kSiteBatchScore)) p.scores[t.out0] = sc;
                p.gathered[tid] = sc;
            }
        }
    }
}

template <bool KEEP>
__global__ void __launch_bounds__(kBandWarps * 32) k_bits_band(BandBitsArgs p) {
    const uint32_t lane = threadIdx.x & 31u;
    for (;;) {
        uint32_t jid = 0;
        if (lane == 0) jid = atomicAdd(p.counter, 1u);
        jid = __shfl_sync(kFull, jid, 0);
        if (jid >= p.njobs) break;
        const BandBitsJob job = p.jobs[jid];
        switch (job.Q) {
            case 1: band_job<1, KEEP>(p, job, lane); break;
            case 2: band_job<2, KEEP>(p, job, lane); break;
            case 3: band_job<3, KEEP>(p, job, lane); break;
            default: band_job<4, KEEP>(p, job, lane); break;
        }
    }
}

// ---------------------------------------------------------------- the walk
struct BitsWalkTask {
    uint64_t ptr_off;         // the pair's first kept planes
    uint64_t moves_off;       // its move bytes
    int64_t a_slot, b_slot;   // planar slots of A (rows) and B (columns)
    uint32_t m, n, gq, Q;
    int32_t hi, a_first;
    uint32_t slot;            // its move count slot
    uint32_t nblocks;
    uint64_t own_off;         // its stretches' moves
    uint64_t rec_off;         // the cells its stretches enter their blocks with, by block
};

// A stretch of a pair's walk: `stretch` blocks, the s-th counted from (m, n).
// The first starts at (m, n), a later one with a cell of the anti-diagonal
// before block c_start; it ends with the first cell before block c_stop.  The
// stretches of a pair follow one another in the table.
struct BitsWalker {
    uint32_t pair, s;
};
struct Stretch {
    int32_t c_start, c_stop;    // c_start: -1 for the first
    bool last;
    uint64_t moves_off, joint_off;  // its moves, and those that lead from its end to the next
    __device__ Stretch(const BitsWalkTask &t, uint32_t s, uint32_t len) {
        c_start = s ? (int32_t)(t.nblocks - s * len) : -1;
        c_stop = max((int32_t)(t.nblocks - (s + 1) * len), 0);
        last = c_stop == 0;
        moves_off = t.own_off + (uint64_t)(2 * s) * stretch_bytes(len);
        joint_off = moves_off + stretch_bytes(len);
    }
    // A move takes one anti-diagonal at least; a copy reads up to 7 bytes beyond.
    __host__ __device__ static uint64_t stretch_bytes(uint32_t len) { return 64ull * len + 32; }
};
// Where a stretch, or the way to the next one, ended (i < 0: outside the
// window), its moves, and the next stretch's moves before the common cell (-1: none).
struct BitsWalkEnd {
    int32_t i, j;
    uint32_t k;
    int32_t joined;
};

// How far a pair's moves are put together: nothing yet; as far as a cell of
// stretch w, its moves after the first `from` to follow; as far as (i, j), from
// where a walk has to look for stretch w or a later one (kNoStretch: for none);
// all.
enum LinkState : uint32_t { kLinkNone, kLinkAt, kLinkLost, kLinkDone };
constexpr uint32_t kNoStretch = ~0u;
struct BitsLink {
    uint32_t state, w, from;
    int32_t i, j;
    uint32_t pad;
    uint64_t moves;
};

struct BitsWalkArgs {
    const uint32_t *pl0, *pl1;
    int64_t max_base;
    const uint4 *ptr;
    const BitsWalkTask *tasks;
    const BitsWalker *walkers;
    uint32_t nwalkers, stretch;
    uint8_t *moves;            // the pairs' moves
    uint64_t *nmoves;
    uint8_t *own;              // the stretches' moves
    int2 *cells;               // first cells of the stretches
    uint4 *recs;               // (i, j, moves so far, 1) of a block entered
    BitsWalkEnd *ends, *joints;
    BitsLink *links;           // per first stretch
    uint32_t last_round;       // lost pairs are walked to their end
    uint32_t half;             // 2^31
    uint64_t moves_cap, own_cap, recs_cap;  // entries at moves, own, recs (checked build)
    uint32_t ntasks;
    uint32_t *err;
};

// The stretches; the ways from the end of each to the next; the walks of pairs
// whose way from one stretch missed the whole next one.
enum WalkMode { kWalkStretches, kWalkJoints, kWalkLost };

// First cells of the later stretches: on the anti-diagonal before their block,
// the cell with the largest W of those inside the grid (the first of several):
// W falls off quickly to either side of the best path.  One warp per stretch;
// W along the anti-diagonal from the kept planes, 32 rows a lane: down one row
// adds that cell's dV and takes off the dH of the cell above it.
__global__ void k_bits_peaks(BitsWalkArgs p) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t wi = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; wi < p.nwalkers;
         wi += (gridDim.x * blockDim.x) >> 5) {
        const BitsWalker wr = p.walkers[wi];
        if (!wr.s) continue;
        const BitsWalkTask tk = p.tasks[wr.pair];
        const Stretch wk(tk, wr.s, p.stretch);
        const int32_t R = (tk.a_first - tk.hi - 1) >> 1, r0 = R + 32 * wk.c_start, a = tk.a_first + 64 * wk.c_start - 1;
        const uint4 *kept = p.ptr + tk.ptr_off + (uint64_t)(wk.c_start / kBlockChunks) * tk.gq;
        int32_t base = 0;                           // W before the words at work
        uint32_t h0_in = 0, h1_in = 0;              // the last dH bits of the words before
        int32_t best = INT_MIN, best_P = -1;
        for (uint32_t w0 = 0; w0 < tk.gq; w0 += 32) {
            const uint32_t wd = w0 + lane;
            uint32_t H0 = 0, H1 = 0, V0 = 0, V1 = 0;
            if (wd < tk.gq) {
                const uint32_t first = wd / tk.Q * tk.Q;
                uint32_t x[4][kBandBitsMaxQ];
#pragma unroll
                for (int v = 0; v < kBandBitsMaxQ; ++v) {
                    const uint4 h = v < (int)tk.Q ? __ldcg(kept + first + v) : make_uint4(0u, 0u, 0u, 0u);
                    x[0][v] = h.x;
                    x[1][v] = h.y;
                    x[2][v] = h.z;
                    x[3][v] = h.w;
                }
                H0 = collect_rows(x[0], tk.Q, wd - first);
                H1 = collect_rows(x[1], tk.Q, wd - first);
                V0 = collect_rows(x[2], tk.Q, wd - first);
                V1 = collect_rows(x[3], tk.Q, wd - first);
            }
            uint32_t c0 = __shfl_up_sync(kFull, H0, 1), c1 = __shfl_up_sync(kFull, H1, 1);
            if (lane == 0) {
                c0 = h0_in;
                c1 = h1_in;
            }
            h0_in = __shfl_sync(kFull, H0, 31);
            h1_in = __shfl_sync(kFull, H1, 31);
            const uint32_t D0 = __funnelshift_l(c0, H0, 1), D1 = __funnelshift_l(c1, H1, 1);  // dH of the cell above
            const int32_t sum = __popc(V0) + 2 * __popc(V1) - __popc(D0) - 2 * __popc(D1);
            int32_t incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t x = __shfl_up_sync(kFull, incl, o);
                if ((int)lane >= o) incl += x;
            }
            int32_t W = base + incl - sum;
            base += __shfl_sync(kFull, incl, 31);
            if (wd < tk.gq) {
                for (int b = 0; b < 32; ++b) {
                    W += (int32_t)((V0 >> b) & 1u) + 2 * (int32_t)((V1 >> b) & 1u) - (int32_t)((D0 >> b) & 1u) -
                         2 * (int32_t)((D1 >> b) & 1u);
                    const int32_t P = 32 * (int32_t)wd + b, i = r0 + P, j = a - i;
                    if (W > best && i >= 1 && j >= 1 && i <= (int32_t)tk.m && j <= (int32_t)tk.n) {
                        best = W;
                        best_P = P;
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const int32_t x = __shfl_xor_sync(kFull, best, o), xP = __shfl_xor_sync(kFull, best_P, o);
            if (xP >= 0 && (best_P < 0 || x > best || (x == best && xP < best_P))) {
                best = x;
                best_P = xP;
            }
        }
        if (lane == 0) p.cells[wi] = best_P < 0 ? make_int2(-1, -1) : make_int2(r0 + best_P, a - r0 - best_P);
    }
}

// A pair's moves from its stretches: each from the cell where the way from the
// one before joined it.  One warp per pair.
__global__ void k_bits_link(BitsWalkArgs p) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t h = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; h < p.nwalkers; h += (gridDim.x * blockDim.x) >> 5) {
        const BitsWalker wr = p.walkers[h];
        if (wr.s) continue;
        const BitsWalkTask tk = p.tasks[wr.pair];
        BitsLink l = p.links[h];
        if (tk.nblocks <= p.stretch || l.state > kLinkAt) continue;
        uint8_t *dst = p.moves + tk.moves_off;
        const uint64_t dst_cap = min(cap_from(tk.moves_off, p.moves_cap), (uint64_t)tk.m + tk.n);
        if (l.state == kLinkNone) l = BitsLink{kLinkAt, h, 0u, (int32_t)tk.m, (int32_t)tk.n, 0u, 0ull};
        l.state = kLinkLost;  // unless the end is reached
        for (uint32_t w = l.w;; ++w) {
            const Stretch wk(tk, w - h, p.stretch);
            const BitsWalkEnd e = p.ends[w];
            l.w = kNoStretch;
            if (e.i < 0) break;
            if (!in_range(l.moves + (e.k - l.from), dst_cap + 1, p.err, kSiteWalkMoves)) break;
            copy_bytes(dst + l.moves, p.own + wk.moves_off + l.from, e.k - l.from, lane, 32);
            l.moves += e.k - l.from;
            l.i = e.i;
            l.j = e.j;
            if (wk.last || e.i == 0 || e.j == 0) {
                l.state = kLinkDone;
                break;
            }
            const BitsWalkEnd x = p.joints[w];
            if (x.i < 0) break;
            if (!in_range(l.moves + x.k, dst_cap + 1, p.err, kSiteWalkMoves)) break;
            copy_bytes(dst + l.moves, p.own + wk.joint_off, x.k, lane, 32);
            l.moves += x.k;
            l.i = x.i;
            l.j = x.j;
            if (x.joined < 0) {
                l.w = w + 2;
                if (x.i == 0 || x.j == 0) l.state = kLinkDone;
                break;
            }
            l.from = (uint32_t)x.joined;
        }
        if (l.state == kLinkDone) {
            const uint32_t rest = (uint32_t)(max(l.i, 0) + max(l.j, 0));
            for (uint32_t q = lane; q < rest; q += 32)
                if (in_range(l.moves + q, dst_cap, p.err, kSiteWalkMoves)) dst[l.moves + q] = l.i > 0 ? 1 : 2;
            if (lane == 0 && in_range(tk.slot, p.ntasks, p.err, kSiteWalkEnds)) p.nmoves[tk.slot] = l.moves + rest;
        }
        if (lane == 0) p.links[h] = l;
    }
}

// Eight walks per warp, one per group of 4 lanes.  A group takes the block of
// its cell, places its sub-window of 4 words (128 rows) around the cell's row,
// starts from the planes kept at the block's start (collected from the fill's
// dealt words) and recomputes the block's anti-diagonals up to its own, their
// pointer records into shared memory; then it walks.  A diagonal move keeps
// the cell's row in the window (same word and bit) and goes one record back,
// so a lane reads four of the next 16 cells; their L bits, put together across
// the group, give the run's length, its zero bytes are stored at once, and the
// Hb bit of the cell that ends it gives the vertical or horizontal move.  Moves
// are written in walk order (0 diagonal, 1 vertical, 2 horizontal), as the
// CIGAR assembly reads.
//
// What bounds it: the chain of a block's anti-diagonals (a shuffle, a shift
// and three logic operations each), at 8 to 15% of the issue slots while a
// pair was one walk (10,000 pairs of 2-20 kb, both rounds: 5.4 ms with blocks
// of 128 anti-diagonals and 4 pairs a warp).  In stretches, with blocks of 64
// (65 rows around the path instead of 129, so half the lanes, records and
// instructions a pair), 3.6 ms.
//
// Why recompute: the pointer records of a whole window are 0.25 bytes per
// cell, which bounded the fill by HBM (10,000 pairs of 2-20 kb: 149 GB, 22 ms
// at the measured copy rate, 36 ms measured with them), while the sub-window
// is a small part of the window and its records never leave the SM.
template <int MODE>
__global__ void __launch_bounds__(32) k_bits_walk(BitsWalkArgs p) {
    extern __shared__ uint4 tiles[];  // [group][record of the block][word]
    const uint32_t lane = threadIdx.x, grp = lane / kSubWords, gl = lane % kSubWords;
    uint4 *tile = tiles + grp * kTileRecs;
    for (uint32_t w0 = blockIdx.x * kSubPairs; w0 < p.nwalkers; w0 += gridDim.x * kSubPairs) {
        const uint32_t wi = min(w0 + grp, p.nwalkers - 1);
        const BitsWalker wr = p.walkers[wi];
        const BitsWalkTask tk = p.tasks[wr.pair];
        const Stretch wk(tk, wr.s, p.stretch);
        bool mine = w0 + grp < p.nwalkers;
        if constexpr (MODE == kWalkJoints) mine = mine && !wk.last;
        BitsLink link{};
        if constexpr (MODE == kWalkLost) {
            if (mine = mine && !wr.s && !wk.last; mine) {
                link = p.links[wi];
                mine = link.state == kLinkLost;
            }
        }
        if (!__any_sync(kFull, mine)) continue;
        // a walk from a cell of the pair's path leaves its moves in their place
        const bool whole = MODE == kWalkLost || (MODE == kWalkStretches && wk.c_start < 0 && wk.last);
        int2 cell = make_int2((int32_t)tk.m, (int32_t)tk.n);
        int32_t c_stop = MODE == kWalkLost ? 0 : wk.c_stop;
        if constexpr (MODE == kWalkStretches)
            if (wk.c_start >= 0) cell = p.cells[wi];
        uint32_t next = kNoStretch;  // the stretch looked for
        const auto look_for = [&](uint32_t w) {
            next = w;
            c_stop = Stretch(tk, wr.s + (w - wi), p.stretch).c_stop;
        };
        if (mine) {
            if constexpr (MODE == kWalkJoints) {
                const BitsWalkEnd e = p.ends[wi];
                cell = make_int2(e.i, e.j);
                look_for(wi + 1);
            }
            if constexpr (MODE == kWalkLost) {
                cell = make_int2(link.i, link.j);
                if (!p.last_round && link.w != kNoStretch) look_for(link.w);
            }
        }
        const int32_t gq = (int32_t)tk.gq, nw = min(gq, kSubWords);
        const int32_t R = (tk.a_first - tk.hi - 1) >> 1;
        const BandBases bs{p.pl0, p.pl1, p.max_base, tk.a_slot, tk.b_slot};
        const uint32_t nzt = gl == 0 ? 0u : 1u, nzb = (int32_t)gl >= nw - 1 ? 0u : 1u;
        const uint64_t own_at = MODE == kWalkJoints ? wk.joint_off : wk.moves_off;
        uint8_t *mv = whole ? p.moves + tk.moves_off + link.moves : p.own + own_at;
        // moves that fit there (checked build): the pair's, or a stretch's
        const uint64_t mv_cap = whole ? min(cap_from(tk.moves_off + link.moves, p.moves_cap), (uint64_t)tk.m + tk.n - link.moves)
                                      : min(cap_from(own_at, p.own_cap), Stretch::stretch_bytes(p.stretch));
        int32_t a_stop = tk.a_first + 64 * c_stop;  // cells before it are not this walk's
        int32_t i = mine ? cell.x : 0, j = mine ? cell.y : 0, joined = -1;
        uint32_t k = 0;
        // A block's inputs: the kept planes and, for each of its chunks and
        // one more, the lane's A and B words.  The next block's are loaded
        // while this one is computed, for the same sub-window.
        struct Block {
            uint4 h[kBandBitsMaxQ];  // the words of the fill's lane that hold this lane's rows
            uint2 A[kBlockChunks + 1], B[kBlockChunks + 1];
        };
        // (`after`: the block after it at the same sub-window, whose bases overlap)
        auto load = [&](Block &blk, int32_t c0, int32_t ws, const Block *after) {
            const int32_t as = tk.a_first + 64 * c0, r = R + 32 * c0 + 32 * (ws + (int32_t)gl);
            const uint32_t first = (uint32_t)(ws + (int32_t)gl) / tk.Q * tk.Q;
#pragma unroll
            for (int v = 0; v < kBandBitsMaxQ; ++v)
                blk.h[v] = c0 > 0 && (int32_t)gl < nw && v < (int)tk.Q
                               ? __ldcg(p.ptr + tk.ptr_off + (uint64_t)(c0 / kBlockChunks) * gq + first + v)
                               : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int c = 0; c <= kBlockChunks; ++c) {
                blk.A[c] = after && c == kBlockChunks ? after->A[0] : bs.rows(r + 32 * c);
                blk.B[c] = after && c == kBlockChunks ? after->B[0] : bs.cols(as - 1 - r + 32 * c);
            }
        };
        Block cur, ahead;
        int32_t ahead_c0 = -1, ahead_ws = 0;
        // every round makes a move in each walking group or ends its walk
        const auto walking = [&] {
            if constexpr (MODE == kWalkLost) {
                // past the whole stretch: the one after it
                if (joined < 0 && i > 0 && j > 0 && i + j < a_stop) {
                    look_for(next + 1);
                    a_stop = tk.a_first + 64 * c_stop;
                }
            }
            return joined < 0 && i > 0 && j > 0 && i + j >= a_stop;
        };
        for (bool on; __any_sync(kFull, on = walking());) {
            const int32_t a = i + j, P = i - ((a - tk.hi) >> 1), wd = P >> 5;
            if (on && (P < 0 || wd >= gq)) {
                // the walk left the window, which a certified band excludes
                // from (m, n), but not from a first cell off the path
                if (whole && gl == 0) raise_error(p.err, NW_ERR_ARG, 0x50000u + wr.pair);
                i = j = whole ? 0 : -1;
                on = false;
            }
            const int32_t cc = on ? (a - tk.a_first) >> 6 : 0, c0 = cc - cc % kBlockChunks;
            if constexpr (MODE == kWalkStretches) {
                if (on && wk.c_start >= 0 && gl == 0 &&
                    in_range(tk.rec_off + (uint64_t)c0, p.recs_cap, p.err, kSiteWalkRecs))
                    p.recs[tk.rec_off + (uint64_t)c0] = make_uint4((uint32_t)i, (uint32_t)j, k, 1u);
            }
            if constexpr (MODE != kWalkStretches) {
                // the next stretch came through this cell: from here on its moves
                if (on && next != kNoStretch) {
                    const uint4 x = __ldcg(p.recs + tk.rec_off + (uint64_t)c0);
                    if (x.w == 1u && x.x == (uint32_t)i && x.y == (uint32_t)j) {
                        joined = (int32_t)x.z;
                        on = false;
                    }
                }
            }
            int32_t ws = on ? min(max(wd - ((P & 31) < 16 ? kSubWords / 2 : kSubWords / 2 - 1), 0), max(gq - kSubWords, 0)) : 0;
            // the words loaded ahead, when the path's rows lie far enough inside them
            const bool hit = on && c0 == ahead_c0 && (ahead_ws == 0 || P - 32 * ahead_ws > kBlockSteps) &&
                             (ahead_ws + kSubWords >= gq || P - 32 * ahead_ws < 32 * kSubWords - 1 - kBlockSteps);
            if (hit) {
                ws = ahead_ws;
                cur = ahead;
            }
            if (on && !hit) load(cur, c0, ws, nullptr);
            ahead_c0 = on ? c0 - kBlockChunks : -1;
            ahead_ws = ws;
            if (ahead_c0 >= c_stop) load(ahead, ahead_c0, ahead_ws, &cur);
            else ahead_c0 = -1;
            const int32_t as = tk.a_first + 64 * c0, r0 = R + 32 * c0 + 32 * ws;  // the block's first step, its top row
            BandWords<1> w;
            {
                const uint32_t word = (uint32_t)(ws + (int32_t)gl), part = word % tk.Q;
                uint32_t x[4][kBandBitsMaxQ];
#pragma unroll
                for (int v = 0; v < kBandBitsMaxQ; ++v) {
                    x[0][v] = cur.h[v].x;
                    x[1][v] = cur.h[v].y;
                    x[2][v] = cur.h[v].z;
                    x[3][v] = cur.h[v].w;
                }
                w.H0[0] = collect_rows(x[0], tk.Q, part);
                w.H1[0] = collect_rows(x[1], tk.Q, part);
                w.V0[0] = collect_rows(x[2], tk.Q, part);
                w.V1[0] = collect_rows(x[3], tk.Q, part);
            }
            __syncwarp();
#pragma unroll
            for (int32_t c = 0; c < kBlockChunks; ++c) {
                const bool live = on && c0 + c <= cc;
                if (!__any_sync(kFull, live)) break;
                const int32_t rc = r0 + 32 * c, ac = as + 64 * c;
                w.A0[0] = cur.A[c].x;
                w.A1[0] = cur.A[c].y;
                w.inA0 = cur.A[c + 1].x;
                w.inA1 = cur.A[c + 1].y;
                w.B0[0] = cur.B[c].x;
                w.B1[0] = cur.B[c].y;
                w.inB0 = cur.B[c + 1].x;
                w.inB1 = cur.B[c + 1].y;
                const bool ramp = __any_sync(kFull, live && !(rc >= 1 && ac - rc - 32 * nw >= 0));
                uint4 *out = tile + 32 * c * kSubWords + gl;
                auto steps = [&](auto ramp_tag) {
                    band_chunk<1>(w, [&](int d, auto) {
                        band_two<1, 0, decltype(ramp_tag)::value, true>(
                            w, kSubWords, nzt, nzb, p.half, rc + d + 32 * (int32_t)gl, ac - rc + d - 32 * (int32_t)gl,
                            [](uint32_t, uint32_t) {},
                            [&](int, uint32_t Ln, uint32_t Hn, uint32_t Ls, uint32_t Hs) {
                                out[d * kSubWords] = make_uint4(Ln, Hn, Ls, Hs);
                            });
                    });
                };
                if (ramp) steps(std::true_type{});
                else steps(std::false_type{});
            }
            __syncwarp();
            // the walk through the block's records
            while (__any_sync(kFull, on)) {
                const int32_t a2 = i + j, rel = a2 - as, x = rel >> 1, par = rel & 1;
                const int32_t P2 = i - ((a2 - tk.hi) >> 1), y = (P2 >> 5) - ws;
                // (a block's path stays within its sub-window; the window's own ends are checked above)
                on = on && rel >= 0 && i > 0 && j > 0 && P2 >= 0 && y >= 0 && y < nw;
                const uint32_t bit = (uint32_t)P2 & 31u;
                // the L bits of the 16 cells from here on along the diagonal in
                // the low half, their Hb bits in the high half; cells outside
                // the block end the run
                uint32_t bits = 0u;
                if (on) {
                    const uint2 *col = reinterpret_cast<const uint2 *>(tile + y) + par;
#pragma unroll
                    for (int q = 0; q < kAhead; ++q) {
                        const int32_t xq = x - kAhead * (int32_t)gl - q;
                        const uint2 rc = xq >= 0 ? col[xq * (2 * kSubWords)] : make_uint2(~0u, 0u);
                        bits |= ((rc.x >> bit) & 1u) << q | ((rc.y >> bit) & 1u) << (16 + q);
                    }
                    bits <<= kAhead * gl;
                }
#pragma unroll
                for (int o = 1; o < kSubWords; o <<= 1) bits |= __shfl_xor_sync(kFull, bits, o);
                if (on) {
                    const uint32_t stop = bits & 0xFFFFu, hb = bits >> 16;
                    const int32_t fr = stop ? __ffs(stop) - 1 : 16;
                    const int32_t run = min(fr, min(i, j));
#pragma unroll
                    for (int q = 0; q < kAhead; ++q)
                        if ((int32_t)gl + kSubWords * q < run &&
                            in_range(k + gl + kSubWords * q, mv_cap, p.err, kSiteWalkMoves))
                            mv[k + gl + kSubWords * q] = 0;
                    k += (uint32_t)run;
                    i -= run;
                    j -= run;
                    if (run == fr && fr < 16 && x - fr >= 0 && i > 0 && j > 0) {
                        const uint32_t mvc = ((hb >> fr) & 1u) ? 2u : 1u;
                        if (gl == 0 && in_range(k, mv_cap, p.err, kSiteWalkMoves)) mv[k] = (uint8_t)mvc;
                        ++k;
                        i -= mvc == 1u;
                        j -= mvc == 2u;
                    }
                }
            }
            __syncwarp();
        }
        if (mine && !whole) {
            if (gl == 0 && in_range(wi, p.nwalkers, p.err, kSiteWalkEnds)) (MODE == kWalkJoints ? p.joints : p.ends)[wi] = BitsWalkEnd{i, j, k, joined};
        } else if (mine && joined >= 0) {
            if (gl == 0 && in_range(wi, p.nwalkers, p.err, kSiteWalkEnds)) p.links[wi] = BitsLink{kLinkAt, next, (uint32_t)joined, i, j, 0u, link.moves + k};
        } else if (mine) {
            // row 0 / column 0: only horizontal / vertical moves remain
            const uint32_t rest = (uint32_t)(max(i, 0) + max(j, 0));
            const uint8_t mvr = i > 0 ? 1 : 2;
            for (uint32_t q = gl; q < rest; q += kSubWords)
                if (in_range(k + q, mv_cap, p.err, kSiteWalkMoves)) mv[k + q] = mvr;
            if (gl == 0 && in_range(tk.slot, p.ntasks, p.err, kSiteWalkEnds)) p.nmoves[tk.slot] = link.moves + k + rest;
            if (MODE == kWalkLost && gl == 0) p.links[wi].state = kLinkDone;
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ host
static uint32_t next_pow2(uint32_t x) {
    uint32_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

int band_bits_max_q() {
    const char *e = getenv("NW_BBAND_MAXQ");
    const int q = e ? atoi(e) : 0;
    return q >= 1 && q <= kBandBitsMaxQ ? q : kBandBitsMaxQ;
}

bool band_bits_shape(uint32_t m, uint32_t n, int32_t lo, int32_t hi, BandBitsShape *s, int max_q) {
    const int32_t hip = hi + (int32_t)(((int64_t)m + n - hi) & 1);
    const int64_t words = ((int64_t)hip - lo + 4 + 63) / 64;
    if (words > kBandBitsMaxWords) return false;
    // throughput shape: the fewest lanes with at most max_q words each (a
    // lane's fixed work per step is shared by more words)
    max_q = std::min(std::max(max_q, 1), kBandBitsMaxQ);
    s->g = std::min<uint32_t>(32, next_pow2((uint32_t)((words + max_q - 1) / max_q)));
    s->Q = (uint32_t)((words + s->g - 1) / s->g);
    s->words = (uint32_t)words;
    s->hi = hip;
    s->nchunks = (uint32_t)(((uint64_t)m + n + 1 + 63) / 64);
    s->a_first = (int32_t)((int64_t)m + n + 1 - 64 * (int64_t)s->nchunks);
    return true;
}

bool band_bits_spread(BandBitsShape *s) {
    if (s->g == 32 || s->Q == 1) return false;
    s->g *= 2;
    s->Q = (s->words + s->g - 1) / s->g;
    return true;
}

uint32_t band_bits_max_width(uint32_t m, uint32_t n) {
    // 2w + |n-m| + 5 <= 64 * kBandBitsMaxWords covers the parity raise of hi
    const int64_t d = (int64_t)n - (int64_t)m, ad = d < 0 ? -d : d;
    const int64_t w = (64 * (int64_t)kBandBitsMaxWords - ad - 5) / 2;
    return w > 0 ? (uint32_t)w : 0u;
}

uint64_t band_bits_cells(const BandBitsShape &s) { return (uint64_t)s.nchunks * 64u * 32u * s.g * s.Q; }

uint64_t band_bits_kept(const BandBitsShape &s) {
    return (uint64_t)((s.nchunks + kBlockChunks - 1) / kBlockChunks) * s.g * s.Q;
}

uint64_t band_bits_scratch(uint32_t m, uint32_t n, const BandBitsShape &s) {
    return band_bits_kept(s) * 16 + m + n + 16 + sizeof(BandBitsTask) + sizeof(BandBitsJob) + sizeof(BitsWalkTask) +
           sizeof(TraceTask) + sizeof(uint64_t) + 4 + (s.nchunks / kStretch + 1) * sizeof(BitsWalker);
}

double band_bits_seconds(const BandBitsShape &s) {
    // 32 pairs of anti-diagonals per chunk, 20 instructions per word and 14
    // per lane each, 2.1 cycles apiece on a scheduler of its own, 2 GHz
    return (double)s.nchunks * 32.0 * (20.0 * s.Q + 14.0) * 2.1 / 2.0e9;
}

int band_bits_fill(nw_ctx *ctx, const PlaneSet &planes, const std::vector<BandBitsItem> &items, bool want, int32_t gap, int32_t *scores, uint32_t score_cap,
                   void *ptr, uint64_t kept, std::vector<int32_t> &banded) {
    int rc;
    banded.assign(items.size(), 0);
    if (items.empty()) return NW_OK;
    HostTimer ht(ctx, "bband_fill_host");
    HostTimer htp(ctx, "bband_fill_prep");
    // jobs: pairs of equal shape (g, Q), similar lengths, 32/g per warp
    // (Q, g, chunks), each descending, ties in item order
    std::vector<uint64_t> keys(items.size());
    for (size_t k = 0; k < items.size(); ++k) {
        const BandBitsShape &sh = items[k].shape;
        keys[k] = ((uint64_t)sh.Q << 40) | ((uint64_t)sh.g << 32) | sh.nchunks;
    }
    const std::vector<uint32_t> order = radix_order_desc(std::move(keys));
    std::vector<BandBitsTask> tasks(items.size());
    std::vector<uint32_t> task_item(items.size());
    std::vector<BandBitsJob> jobs;
    for (uint32_t k = 0; k < order.size();) {
        const BandBitsShape &s0 = items[order[k]].shape;
        BandBitsJob j{k, 0, s0.g, s0.Q, s0.nchunks};
        while (k < order.size() && j.cnt < 32 / s0.g && items[order[k]].shape.g == s0.g &&
               items[order[k]].shape.Q == s0.Q) {
            const BandBitsItem &it = items[order[k]];
            BandBitsTask &t = tasks[k];
            t.a_slot = it.a_slot;
            t.b_slot = it.b_slot;
            t.ptr_off = it.ptr_off;
            t.m = it.m;
            t.n = it.n;
            t.hi = it.shape.hi;
            t.a_first = it.shape.a_first;
            t.nchunks = it.shape.nchunks;
            t.out0 = it.out0;
            task_item[k] = order[k];
            ++j.cnt;
            ++k;
        }
        jobs.push_back(j);
    }
    // longest jobs first (ties in job order)
    double work = 0, longest = 0;
    {
        std::vector<uint64_t> jk(jobs.size());
        for (size_t q = 0; q < jobs.size(); ++q) {
            jk[q] = (uint64_t)jobs[q].nchunks * (20 * jobs[q].Q + 14);
            work += (double)jk[q];
            longest = std::max(longest, (double)jk[q]);
        }
        const std::vector<uint32_t> jo = radix_order_desc(std::move(jk));
        std::vector<BandBitsJob> sorted(jobs.size());
        for (size_t q = 0; q < jobs.size(); ++q) sorted[q] = jobs[jo[q]];
        jobs.swap(sorted);
    }
    void *v = nullptr;
    if ((rc = scratch(ctx, "bband_tasks", tasks.size() * sizeof(BandBitsTask) + 16, &v))) return rc;
    BandBitsTask *dt = (BandBitsTask *)v;
    if ((rc = scratch(ctx, "bband_jobs", jobs.size() * sizeof(BandBitsJob) + 16, &v))) return rc;
    BandBitsJob *dj = (BandBitsJob *)v;
    if ((rc = scratch(ctx, "bband_gather", items.size() * 4 + 16, &v))) return rc;
    int32_t *dg = (int32_t *)v;
    if ((rc = scratch(ctx, "bband_counter", 16, &v))) return rc;
    uint32_t *cnt = (uint32_t *)v;
    cudaError_t e = cudaMemcpyAsync(dt, tasks.data(), tasks.size() * sizeof(BandBitsTask), cudaMemcpyHostToDevice,
                                    ctx->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dj, jobs.data(), jobs.size() * sizeof(BandBitsJob), cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, 4, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "banded bit-sliced tasks H2D");
    BandBitsArgs a{};
    a.pl0 = planes.pl0;
    a.pl1 = planes.pl1;
    a.max_base = planes.max_base;
    a.tasks = dt;
    a.jobs = dj;
    a.njobs = (uint32_t)jobs.size();
    a.counter = cnt;
    a.ptr = (uint4 *)ptr;
    a.ptr_cap = kept;
    a.scores = scores;
    a.gathered = dg;
    a.score_cap = score_cap;
    a.gap = gap;
    a.two = 2u;
    a.half = 1u << 31;
    a.err = ctx->d_err;
    auto kern = want ? k_bits_band<true> : k_bits_band<false>;
    htp.stop();
    // Two CTAs per SM (two warps per scheduler), not the most the registers
    // allow: the jobs are taken longest first, and a long job that shares its
    // scheduler with others ends the launch alone.  One CTA where even beside
    // one other the longest job would outlast the launch's ideal time (every
    // scheduler busy).  Fills of both rounds on GB300, pairs of 2-20 kb, one /
    // two CTAs: 2,500 pairs 4.4 / 6.9 ms, 10,000 pairs 10.3 / 10.9 ms, 20,000
    // pairs 20.5 / 18.0 ms.  NW_BBAND_OCC overrides (sweeps).
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kBandWarps * 32, 0);
    int cap = 2.0 * longest > work / (4.0 * ctx->sm_count) ? 1 : 2;
    if (const char *e = getenv("NW_BBAND_OCC")) cap = std::max(1, atoi(e));
    occ = std::min(occ, cap);
    uint32_t blocks = (uint32_t)std::max(occ, 1) * (uint32_t)ctx->sm_count;
    blocks = std::max(1u, std::min(blocks, (a.njobs + kBandWarps - 1) / kBandWarps));
    {
        LaunchTimer t(ctx, want ? "bband_fill_ptr" : "bband_score");
        kern<<<blocks, kBandWarps * 32, 0, ctx->stream>>>(a);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(ctx, e, "banded bit-sliced launch");
    // the banded scores back, in item order
    std::vector<int32_t> g(items.size());
    e = cudaMemcpyAsync(g.data(), dg, items.size() * 4, cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "banded scores D2H");
    {
        HostTimer ht(ctx, "band_wait");
        if ((rc = nw_ctx_sync(ctx))) return rc;
    }
    for (size_t k = 0; k < items.size(); ++k) banded[task_item[k]] = g[k];
    return NW_OK;
}

int band_bits_walk(nw_ctx *ctx, const PlaneSet &planes, const void *ptr, const std::vector<BandBitsItem> &items,
                   const std::vector<uint32_t> &which, const uint8_t *pool, char *cigar_pool,
                   const uint64_t *cigar_off, uint64_t *cigar_len, uint32_t mflag) {
    if (which.empty()) return NW_OK;
    int rc;
    HostTimer ht(ctx, "bband_walk_host");
    // longest walks first: the kernel's warps take pairs in order
    std::vector<uint32_t> order(which.size());
    {
        std::vector<uint64_t> wk(which.size());
        for (size_t q = 0; q < which.size(); ++q) wk[q] = (uint64_t)items[which[q]].m + items[which[q]].n;
        const std::vector<uint32_t> wo = radix_order_desc(std::move(wk));  // ties in `which` order
        for (size_t q = 0; q < which.size(); ++q) order[q] = which[wo[q]];
    }
    uint64_t mbytes = 0;
    for (uint32_t k : order) mbytes += (uint64_t)items[k].m + items[k].n + 16;
    void *mv = nullptr, *nm = nullptr, *v = nullptr;
    if ((rc = scratch(ctx, "bband_moves", mbytes + 16, &mv))) return rc;
    if ((rc = scratch(ctx, "bband_nmoves", which.size() * 8 + 16, &nm))) return rc;
    std::vector<BitsWalkTask> wt(which.size());
    std::vector<TraceTask> tt(which.size());
    uint64_t mpos = 0;
    for (size_t q = 0; q < order.size(); ++q) {
        const BandBitsItem &it = items[order[q]];
        wt[q] = BitsWalkTask{it.ptr_off, mpos, it.a_slot, it.b_slot, it.m, it.n, it.shape.g * it.shape.Q, it.shape.Q, it.shape.hi,
                             it.shape.a_first, (uint32_t)q, it.shape.nchunks / kBlockChunks, 0, 0};
        static_assert(kBlockChunks == 1, "nblocks");
        TraceTask x{};
        x.m = it.m;
        x.n = it.n;
        x.moves = (uint8_t *)mv + mpos;
        x.nmoves = (uint64_t *)nm + q;
        x.a = pool + it.a_off;
        x.b = pool + it.b_off;
        x.cigar = cigar_pool + cigar_off[it.out0];
        x.cigar_len = cigar_len + it.out0;
        x.band_lo = kNoBand;
        tt[q] = x;
        mpos += (uint64_t)it.m + it.n + 16;
    }
    if ((rc = scratch(ctx, "bband_walk_tasks", wt.size() * sizeof(BitsWalkTask) + 16, &v))) return rc;
    BitsWalkTask *dw = (BitsWalkTask *)v;
    // Whole pairs where the stretches' moves and records would take more than a
    // quarter of the scratch that is left.  NW_BBAND_STRETCH: blocks of a
    // stretch (sweeps, tests).
    uint32_t len = kStretch;
    if (const char *e = getenv("NW_BBAND_STRETCH")) len = (uint32_t)std::max(1, atoi(e));
    uint64_t own = 0, recs = 0, nwalkers = 0;
    for (BitsWalkTask &t : wt) {
        const uint32_t segs = (t.nblocks + len - 1) / len;
        t.own_off = own;
        t.rec_off = recs;
        nwalkers += segs;
        if (segs == 1) continue;
        own += 2 * segs * Stretch::stretch_bytes(len);
        recs += t.nblocks;
    }
    const uint64_t extra =
        nwalkers * (sizeof(int2) + 2 * sizeof(BitsWalkEnd) + sizeof(BitsLink)) + recs * sizeof(uint4) + own + 64;
    bool split = nwalkers > wt.size();
    if (split && extra > scratch_headroom(ctx, "bband_stretch") / 4) {
        split = false;
        len = 1u << 30;
    }
    std::vector<BitsWalker> wk;
    wk.reserve(nwalkers);
    for (size_t q = 0; q < wt.size(); ++q)
        for (uint32_t s = 0; (uint64_t)s * len < wt[q].nblocks; ++s) wk.push_back(BitsWalker{(uint32_t)q, s});
    if ((rc = scratch(ctx, "bband_walkers", wk.size() * sizeof(BitsWalker) + 16, &v))) return rc;
    BitsWalker *dwk = (BitsWalker *)v;
    if ((rc = scratch(ctx, "bband_trace_tasks", tt.size() * sizeof(TraceTask) + 16, &v))) return rc;
    TraceTask *dtt = (TraceTask *)v;
    cudaError_t e = cudaMemcpyAsync(dw, wt.data(), wt.size() * sizeof(BitsWalkTask), cudaMemcpyHostToDevice,
                                    ctx->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dtt, tt.data(), tt.size() * sizeof(TraceTask), cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dwk, wk.data(), wk.size() * sizeof(BitsWalker), cudaMemcpyHostToDevice, ctx->stream);
    // the host task arrays go out of scope: wait for their copies (the fill
    // before them has finished already; its scores were read back), not for
    // the walk, so the caller prepares its next round while the GPU walks
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "walk tasks H2D");
    BitsWalkArgs wa{};
    wa.pl0 = planes.pl0;
    wa.pl1 = planes.pl1;
    wa.max_base = planes.max_base;
    wa.ptr = (const uint4 *)ptr;
    wa.tasks = dw;
    wa.walkers = dwk;
    wa.nwalkers = (uint32_t)wk.size();
    wa.stretch = len;
    wa.moves = (uint8_t *)mv;
    wa.nmoves = (uint64_t *)nm;
    wa.moves_cap = mbytes;
    wa.own_cap = own;
    wa.recs_cap = recs;
    wa.ntasks = (uint32_t)wt.size();
    wa.half = 1u << 31;
    wa.err = ctx->d_err;
    if (split) {
        if ((rc = scratch(ctx, "bband_stretch", extra, &v))) return rc;
        uint8_t *at = (uint8_t *)v;
        wa.links = (BitsLink *)at;
        at += wk.size() * sizeof(BitsLink);
        wa.recs = (uint4 *)(at + (16 - (uintptr_t)at % 16) % 16);
        at = (uint8_t *)(wa.recs + recs);
        e = cudaMemsetAsync(v, 0, (size_t)(at - (uint8_t *)v), ctx->stream);  // nothing linked, no block entered
        if (e != cudaSuccess) return cuda_fail(ctx, e, "walk records");
        wa.ends = (BitsWalkEnd *)at;
        at += wk.size() * sizeof(BitsWalkEnd);
        wa.joints = (BitsWalkEnd *)at;
        at += wk.size() * sizeof(BitsWalkEnd);
        wa.cells = (int2 *)at;
        at += wk.size() * sizeof(int2);
        wa.own = at;
    }
    {
        LaunchTimer t(ctx, "bband_walk", split ? 7 : 1);  // peaks, stretches, joints, two rounds of link and lost
        // one warp per CTA; its 17 KB of records let 13 share an SM
        constexpr int smem = kSubPairs * kTileRecs * (int)sizeof(uint4);
        static_assert(smem <= 48 * 1024, "above the default limit of dynamic shared memory");
        const uint32_t blocks = (uint32_t)std::min<size_t>((wk.size() + kSubPairs - 1) / kSubPairs, 65535);
        const uint32_t warps = (uint32_t)std::min<size_t>((wk.size() + 7) / 8, 65535);
        if (split) k_bits_peaks<<<warps, 256, 0, ctx->stream>>>(wa);
        k_bits_walk<kWalkStretches><<<blocks, 32, smem, ctx->stream>>>(wa);
        if (split) {
            k_bits_walk<kWalkJoints><<<blocks, 32, smem, ctx->stream>>>(wa);
            for (wa.last_round = 0; wa.last_round < 2; ++wa.last_round) {
                k_bits_link<<<warps, 256, 0, ctx->stream>>>(wa);
                k_bits_walk<kWalkLost><<<blocks, 32, smem, ctx->stream>>>(wa);
            }
        }
    }
    if (split) free_prefix(ctx, "bband_stretch");  // in stream order
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(ctx, e, "walk launch");
    return launch_finish(ctx, TraceTask{}, dtt, (uint32_t)tt.size(), mflag);
}

}  // namespace nw
