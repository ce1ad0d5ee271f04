// Bit-sliced certified band (a8) with pointers (a4) and its walk (a5).
//
// The fill is the difference form of nw_bits.cu (dH, dV in two bit planes,
// T = max(s', a, b), dV = T - a, dH = T - b) on a window that follows the
// band: on anti-diagonal a the window holds the Hw = 32*g*Q rows
// r0(a) .. r0(a)+Hw-1 with r0(a) = floor((a - hi)/2), so it moves down one
// row every second anti-diagonal and always covers the band's diagonals
// [lo, hi] (2*Hw >= hi - lo + 4).  A pair belongs to a group of g lanes
// (1..32, a power of two) holding Q words each; window bit P = 32*(lane*Q +
// word) + bit is row r0(a) + P, column a - r0(a) - P.
//
// Anti-diagonals come in pairs: a step where r0 stays (the B bases slide one
// bit up, a new column enters at the top; the cell above a bit is the bit
// below it on the previous anti-diagonal, the cell to its left the same bit)
// and a step where r0 grows (the A bases slide one bit down, a new row
// enters at the bottom; the cell above is the same bit, the cell to the left
// the bit above).  Shifts across words go through funnel shifts, across
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
// The score is tracked at the window's top cell (its dH on a step without a
// shift, its dV on a shift) and carried down the last anti-diagonal to
// (m, n).
//
// Alignments.  The fill writes no pointers: every kBlockChunks chunks (128
// anti-diagonals) it keeps the window's four planes (16 bytes per word).  The
// walk then goes back block by block: it recomputes the pointer bits of the
// block it stands in from the planes kept at its start -- only the 256 rows
// around the path, because a cell of an anti-diagonal depends on the row
// itself and its two neighbours one anti-diagonal pair earlier, so nothing
// further than 64 rows away reaches the path within 128 anti-diagonals -- into
// shared memory and follows the path through them.  Pointer bits, per cell:
// L = T != s' (the diagonal loses), and Hb = dV != 0 (the vertical move
// loses); the walk reads !L -> diagonal, else !Hb -> vertical, else
// horizontal, the diagonal > vertical > horizontal order of the scalar
// kernels.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <type_traits>
#include <vector>

#include "nw_bits.cuh"
#include "nw_order.h"

namespace nw {

// Words per lane: at most 4, so a pair's window holds up to 128 words (4,096
// rows, bands up to ~8,190 diagonals).  Up to 8 words per lane (fewer lanes
// per pair, the lane's fixed work per step shared by more words) measured
// 1.5x slower on the band workload: 27.3 against 18.0 ms per fill.
constexpr int kBandBitsMaxQ = 4;
constexpr int kBandBitsMaxWords = 32 * kBandBitsMaxQ;
// Anti-diagonals between kept planes: kBlockChunks chunks of 64; the walk's
// sub-window of kSubWords words covers the rows a block's path can depend on.
constexpr int kBlockChunks = 2;
constexpr int kSubWords = 8;
constexpr int kSubPairs = 32 / kSubWords;                // pairs per warp of the walk
constexpr int kBlockSteps = 32 * kBlockChunks;           // pairs of anti-diagonals per block
static_assert(kSubWords * 32 >= 2 * (kBlockSteps + 1) + 16 + 32, "the sub-window must hold a block's dependencies");
// Warps per CTA of the fill: at ~150 registers an SM holds 13 warps, so
// CTAs of 4 warps fit 12 of them (CTAs of 8 only 8).
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

// A lane's Q words of the window: difference planes, the bases of the
// chunk's start, and the words that follow them (in: the word above the
// lane's first for B, below its last for A).  During a chunk the B bases of a
// word slide up by 32 and its A bases down by 32, so both always lie in two
// of these words and a step takes them by one funnel shift; after it each
// word holds what its neighbour held.
template <int Q>
struct BandWords {
    uint32_t A0[Q], A1[Q], B0[Q], B1[Q], H0[Q], H1[Q], V0[Q], V1[Q];
    uint32_t inA0, inA1, inB0, inB1;
    __device__ __forceinline__ void next_chunk() {
        uint32_t a0 = inA0, a1 = inA1, b0 = inB0, b1 = inB1;
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            const uint32_t x0 = B0[v], x1 = B1[v];
            B0[v] = b0;
            B1[v] = b1;
            b0 = x0;
            b1 = x1;
        }
#pragma unroll
        for (int v = Q - 1; v >= 0; --v) {
            const uint32_t x0 = A0[v], x1 = A1[v];
            A0[v] = a0;
            A1[v] = a1;
            a0 = x0;
            a1 = x1;
        }
    }
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

// A pair of anti-diagonals, the d-th of its chunk, of a window spread over
// groups of g lanes.  The first has the lane's first word at row r (bit 0)
// and columns 1 .. at bits below cmax; nzt, nzb: 0 on the group's top /
// bottom lane, else 1.  cA: the A words of the step before, then of this one.
// top() runs after the first with the lane's first H word, after the second
// with its first V word (the score's path); rec(v, L, Hb, L', Hb') takes the
// pointer bits.
//
// What bounds it: the logic pipe, 14 operations per word and anti-diagonal
// (16 with pointers); the choice at the group's ends is a multiply-add,
// which issues beside it.
template <int Q, bool RAMP, bool PTR, class Top, class Rec>
__device__ __forceinline__ void band_two(BandWords<Q> &w, uint32_t (&cA0)[Q], uint32_t (&cA1)[Q], uint32_t d,
                                         uint32_t g, uint32_t nzt, uint32_t nzb, int32_t r, int32_t cmax, Top top,
                                         Rec rec) {
    uint32_t Ln[Q], Hn[Q], cB0[Q], cB1[Q];
    {
        // no shift; above the window a horizontal gap, dH = 0
        const uint32_t sH0 = mul(__shfl_up_sync(kFull, w.H0[Q - 1], 1, g), nzt);
        const uint32_t sH1 = mul(__shfl_up_sync(kFull, w.H1[Q - 1], 1, g), nzt);
#pragma unroll
        for (int v = Q - 1; v >= 0; --v) {
            cB0[v] = __funnelshift_lc(v ? w.B0[v - 1] : w.inB0, w.B0[v], d + 1);
            cB1[v] = __funnelshift_lc(v ? w.B1[v - 1] : w.inB1, w.B1[v], d + 1);
            const uint32_t a0 = __funnelshift_l(v ? w.H0[v - 1] : sH0, w.H0[v], 1);
            const uint32_t a1 = __funnelshift_l(v ? w.H1[v - 1] : sH1, w.H1[v], 1);
            const uint32_t mk = RAMP ? range_mask(1 - r - 32 * v, cmax - 32 * v - 1) : ~0u;
            band_cell<RAMP, PTR>(cA0[v], cA1[v], cB0[v], cB1[v], a0, a1, w.V0[v], w.V1[v], mk, w.H0[v], w.H1[v],
                                 w.V0[v], w.V1[v], Ln[v], Hn[v]);
        }
        top(0, w.H0[0], w.H1[0]);
    }
    {
        // shift; below the window a vertical gap, dV = 0
        const uint32_t sV0 = mul(__shfl_down_sync(kFull, w.V0[0], 1, g), nzb);
        const uint32_t sV1 = mul(__shfl_down_sync(kFull, w.V1[0], 1, g), nzb);
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            cA0[v] = __funnelshift_rc(w.A0[v], v + 1 < Q ? w.A0[v + 1] : w.inA0, d + 1);
            cA1[v] = __funnelshift_rc(w.A1[v], v + 1 < Q ? w.A1[v + 1] : w.inA1, d + 1);
            const uint32_t b0 = __funnelshift_r(w.V0[v], v + 1 < Q ? w.V0[v + 1] : sV0, 1);
            const uint32_t b1 = __funnelshift_r(w.V1[v], v + 1 < Q ? w.V1[v + 1] : sV1, 1);
            const uint32_t mk = RAMP ? range_mask(-r - 32 * v, cmax - 32 * v - 1) : ~0u;
            uint32_t Ls = 0, Hs = 0;
            band_cell<RAMP, PTR>(cA0[v], cA1[v], cB0[v], cB1[v], w.H0[v], w.H1[v], b0, b1, mk, w.H0[v], w.H1[v],
                                 w.V0[v], w.V1[v], Ls, Hs);
            if constexpr (PTR) rec(v, Ln[v], Hn[v], Ls, Hs);
        }
        top(1, w.V0[0], w.V1[0]);
    }
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
#pragma unroll
    for (int v = 0; v < Q; ++v) {
        const uint2 x = bs.rows(R + wo + 32 * v), y = bs.cols(a0 - 1 - R - wo - 32 * v);
        w.A0[v] = x.x;
        w.A1[v] = x.y;
        w.B0[v] = y.x;
        w.B1[v] = y.y;
        w.H0[v] = w.H1[v] = w.V0[v] = w.V1[v] = 0;
    }
    // the bases that enter the window during a chunk, loaded one chunk ahead
    // (the top lane's columns, the bottom lane's rows)
    uint2 fa = bs.rows(R + Hw), fb = bs.cols(a0 - R + 31);
    const uint32_t nzt = gl == 0 ? 0u : 1u, nzb = gl == g - 1 ? 0u : 1u;  // 0 on the group's top / bottom lane
    int32_t top = 0;  // W of the window's top cell
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
        {
            const uint32_t b0 = __shfl_up_sync(kFull, w.B0[Q - 1], 1, g), b1 = __shfl_up_sync(kFull, w.B1[Q - 1], 1, g);
            const uint32_t x0 = __shfl_down_sync(kFull, w.A0[0], 1, g), x1 = __shfl_down_sync(kFull, w.A1[0], 1, g);
            w.inB0 = nzt ? b0 : fb.x;
            w.inB1 = nzt ? b1 : fb.y;
            w.inA0 = nzb ? x0 : fa.x;
            w.inA1 = nzb ? x1 : fa.y;
            fa = bs.rows(rc + 32 + Hw);
            fb = bs.cols(ac + 64 - rc - 32 + 31);
        }
        // masks only while some cell of the chunk lies on or beyond row 0 / column 0
        const bool ramp = __any_sync(kFull, live && !(rc >= 1 && ac - rc - Hw >= 0));
        uint32_t cH0 = 0, cH1 = 0, cV0 = 0, cV1 = 0;
        uint32_t cA0[Q], cA1[Q];
#pragma unroll
        for (int v = 0; v < Q; ++v) {
            cA0[v] = w.A0[v];
            cA1[v] = w.A1[v];
        }
        auto steps = [&](auto ramp_tag) {
            for (int32_t d = 0; d < 32; ++d)
                band_two<Q, decltype(ramp_tag)::value, false>(
                    w, cA0, cA1, (uint32_t)d, g, nzt, nzb, rc + d + wo, ac - rc + d - wo,
                    [&](int second, uint32_t x0, uint32_t x1) {
                        if (!second) {
                            cH0 = __funnelshift_r(cH0, x0, 1);
                            cH1 = __funnelshift_r(cH1, x1, 1);
                        } else {
                            cV0 = __funnelshift_r(cV0, x0, 1);
                            cV1 = __funnelshift_r(cV1, x1, 1);
                        }
                    },
                    [](int, uint32_t, uint32_t, uint32_t, uint32_t) {});
        };
        if (ramp) steps(std::true_type{});
        else steps(std::false_type{});
        w.next_chunk();
        top += __popc(cH0) + 2 * __popc(cH1) + __popc(cV0) + 2 * __popc(cV1);
        if (active && c + 1 == nch) {
            // W(m, n): the top cell, then down the last anti-diagonal: each row
            // adds its cell's dV and takes off the dH of the cell above it
            const int32_t Pm = (int32_t)t.m - (R + 32 * (int32_t)nch);
            int32_t sum = 0;
#pragma unroll
            for (int v = 0; v < Q; ++v) {
                const int32_t o = wo + 32 * v;
                const uint32_t vm = range_mask(1 - o, Pm - o), hm = range_mask(-o, Pm - 1 - o);
                sum += __popc(w.V0[v] & vm) + 2 * __popc(w.V1[v] & vm) - __popc(w.H0[v] & hm) - 2 * __popc(w.H1[v] & hm);
            }
            for (uint32_t o = 1; o < g; o <<= 1) sum += __shfl_xor_sync(gmask, sum, o);
            if (gl == 0) {
                const int32_t sc = top + sum + p.gap * (int32_t)(t.m + t.n);
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
    uint32_t m, n, gq;
    int32_t hi, a_first;
    uint32_t slot;            // its move count slot
};

struct BitsWalkArgs {
    const uint32_t *pl0, *pl1;
    int64_t max_base;
    const uint4 *ptr;
    const BitsWalkTask *tasks;
    uint32_t ntasks;
    uint8_t *moves;
    uint64_t *nmoves;
    uint32_t *err;
};

// Four pairs per warp, one per group of 8 lanes.  A group takes the block of
// its cell, places its sub-window of 8 words (256 rows) around the cell's
// row (at least 65 rows on either side unless the window itself ends),
// starts from the planes kept at the block's start and recomputes the
// block's anti-diagonals up to its own, their pointer records into shared
// memory; then it walks.  A diagonal move keeps the cell's row in the window
// (same word and bit) and goes one record back, so lane t reads the cells t
// and t + 8 diagonal moves on; ballots of their L bits give the run's
// length, its zero bytes are stored at once, and the Hb bit of the cell that
// ends it gives the vertical or horizontal move.  Moves are written in walk
// order (0 diagonal, 1 vertical, 2 horizontal), as the CIGAR assembly reads.
//
// Why recompute: the pointer records of a whole window are 0.25 bytes per
// cell, which bounded the fill by HBM (10,000 pairs of 2-20 kb: 149 GB, 22 ms
// at the measured copy rate, 36 ms measured with them), while the sub-window
// is about a tenth of the window and its records never leave the SM.
__global__ void __launch_bounds__(32) k_bits_walk(BitsWalkArgs p) {
    extern __shared__ uint4 tiles[];  // [group][record of the block][word]
    const uint32_t lane = threadIdx.x, grp = lane / kSubWords, gl = lane % kSubWords;
    uint4 *tile = tiles + grp * (kBlockSteps * kSubWords);
    for (uint32_t w0 = blockIdx.x * kSubPairs; w0 < p.ntasks; w0 += gridDim.x * kSubPairs) {
        const uint32_t ti = w0 + grp;
        const bool mine = ti < p.ntasks;
        const BitsWalkTask tk = p.tasks[mine ? ti : w0];
        const int32_t gq = (int32_t)tk.gq, nw = min(gq, kSubWords);
        const int32_t R = (tk.a_first - tk.hi - 1) >> 1;
        const BandBases bs{p.pl0, p.pl1, p.max_base, tk.a_slot, tk.b_slot};
        const uint32_t nzt = gl == 0 ? 0u : 1u, nzb = (int32_t)gl >= nw - 1 ? 0u : 1u;
        uint8_t *mv = p.moves + tk.moves_off;
        int32_t i = mine ? (int32_t)tk.m : 0, j = mine ? (int32_t)tk.n : 0;
        uint32_t k = 0;
        // A block's inputs: the kept planes and, for each of its chunks and
        // one more, the lane's A and B words.  The next block's are loaded
        // while this one is computed, for the same sub-window.
        struct Block {
            uint4 h;
            uint2 A[kBlockChunks + 1], B[kBlockChunks + 1];
        };
        auto load = [&](Block &blk, int32_t c0, int32_t ws) {
            const int32_t as = tk.a_first + 64 * c0, r = R + 32 * c0 + 32 * (ws + (int32_t)gl);
            blk.h = make_uint4(0u, 0u, 0u, 0u);
            if (c0 > 0 && (int32_t)gl < nw)
                blk.h = __ldcg(p.ptr + tk.ptr_off + (uint64_t)(c0 / kBlockChunks) * gq + ws + gl);
#pragma unroll
            for (int c = 0; c <= kBlockChunks; ++c) {
                blk.A[c] = bs.rows(r + 32 * c);
                blk.B[c] = bs.cols(as - 1 - r + 32 * c);
            }
        };
        Block cur, ahead;
        int32_t ahead_c0 = -1, ahead_ws = 0;
        // every round makes a move in each walking group or ends its walk
        while (__any_sync(kFull, i > 0 && j > 0)) {
            bool on = i > 0 && j > 0;
            const int32_t a = i + j, P = i - ((a - tk.hi) >> 1), wd = P >> 5;
            if (on && (P < 0 || wd >= gq)) {
                // the walk left the window, which a certified band excludes
                if (gl == 0) raise_error(p.err, NW_ERR_ARG, 0x50000u + ti);
                i = j = 0;
                on = false;
            }
            const int32_t cc = on ? (a - tk.a_first) >> 6 : 0, c0 = cc - cc % kBlockChunks;
            int32_t ws = on ? min(max(wd - ((P & 31) < 16 ? 4 : 3), 0), max(gq - kSubWords, 0)) : 0;
            // the words loaded ahead, when the path's rows lie far enough inside them
            const bool hit = on && c0 == ahead_c0 && (ahead_ws == 0 || P - 32 * ahead_ws > kBlockSteps) &&
                             (ahead_ws + kSubWords >= gq || P - 32 * ahead_ws < 32 * kSubWords - 1 - kBlockSteps);
            if (hit) {
                ws = ahead_ws;
                cur = ahead;
            }
            if (on && !hit) load(cur, c0, ws);
            ahead_c0 = on ? c0 - kBlockChunks : -1;
            ahead_ws = ws;
            if (ahead_c0 >= 0) load(ahead, ahead_c0, ahead_ws);
            const int32_t as = tk.a_first + 64 * c0, r0 = R + 32 * c0 + 32 * ws;  // the block's first step, its top row
            BandWords<1> w;
            w.H0[0] = cur.h.x;
            w.H1[0] = cur.h.y;
            w.V0[0] = cur.h.z;
            w.V1[0] = cur.h.w;
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
                uint32_t cA0[1] = {w.A0[0]}, cA1[1] = {w.A1[0]};
                auto steps = [&](auto ramp_tag) {
#pragma unroll 4
                    for (int32_t d = 0; d < 32; ++d)
                        band_two<1, decltype(ramp_tag)::value, true>(
                            w, cA0, cA1, (uint32_t)d, kSubWords, nzt, nzb, rc + d + 32 * (int32_t)gl,
                            ac - rc + d - 32 * (int32_t)gl, [](int, uint32_t, uint32_t) {},
                            [&](int, uint32_t Ln, uint32_t Hn, uint32_t Ls, uint32_t Hs) {
                                out[d * kSubWords] = make_uint4(Ln, Hn, Ls, Hs);
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
                uint32_t L0 = 1u, L1 = 1u, h0 = 0u, h1 = 0u;  // cells outside the block end the run
                if (on) {
                    const int32_t x0 = x - (int32_t)gl, x1 = x0 - kSubWords;
                    if (x0 >= 0) {
                        const uint4 rc = tile[x0 * kSubWords + y];
                        L0 = ((par ? rc.z : rc.x) >> bit) & 1u;
                        h0 = ((par ? rc.w : rc.y) >> bit) & 1u;
                    }
                    if (x1 >= 0) {
                        const uint4 rc = tile[x1 * kSubWords + y];
                        L1 = ((par ? rc.z : rc.x) >> bit) & 1u;
                        h1 = ((par ? rc.w : rc.y) >> bit) & 1u;
                    }
                }
                const uint32_t sh = grp * kSubWords, gm = (1u << kSubWords) - 1u;
                const uint32_t stop = ((__ballot_sync(kFull, L0) >> sh) & gm) |
                                      (((__ballot_sync(kFull, L1) >> sh) & gm) << kSubWords);
                const uint32_t hb = ((__ballot_sync(kFull, h0) >> sh) & gm) |
                                    (((__ballot_sync(kFull, h1) >> sh) & gm) << kSubWords);
                if (on) {
                    const int32_t fr = stop ? __ffs(stop) - 1 : 2 * kSubWords;
                    const int32_t run = min(fr, min(i, j));
                    if ((int32_t)gl < run) mv[k + gl] = 0;
                    if ((int32_t)gl + kSubWords < run) mv[k + gl + kSubWords] = 0;
                    k += (uint32_t)run;
                    i -= run;
                    j -= run;
                    if (run == fr && fr < 2 * kSubWords && x - fr >= 0 && i > 0 && j > 0) {
                        const uint32_t mvc = ((hb >> fr) & 1u) ? 2u : 1u;
                        if (gl == 0) mv[k] = (uint8_t)mvc;
                        ++k;
                        i -= mvc == 1u;
                        j -= mvc == 2u;
                    }
                }
            }
            __syncwarp();
        }
        // row 0 / column 0: only horizontal / vertical moves remain
        if (mine) {
            const uint32_t rest = (uint32_t)(max(i, 0) + max(j, 0));
            const uint8_t mvr = i > 0 ? 1 : 2;
            for (uint32_t q = gl; q < rest; q += kSubWords) mv[k + q] = mvr;
            if (gl == 0) p.nmoves[tk.slot] = (uint64_t)k + rest;
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

void band_bits_fast(BandBitsShape *s) {
    // latency shape: one word per lane while 32 lanes suffice, else 32 lanes
    s->g = std::min<uint32_t>(32, next_pow2(s->words));
    s->Q = (s->words + s->g - 1) / s->g;
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

double band_bits_seconds(const BandBitsShape &s) {
    // 64 anti-diagonals per chunk, ~15 instructions per word and ~10 per
    // lane per step, two cycles each on a scheduler of its own, 2.07 GHz
    return (double)s.nchunks * 64.0 * (15.0 * s.Q + 10.0) * 2.0 / 2.07e9;
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
            jk[q] = (uint64_t)jobs[q].nchunks * (15 * jobs[q].Q + 10);
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
    a.err = ctx->d_err;
    auto kern = want ? k_bits_band<true> : k_bits_band<false>;
    htp.stop();
    // Two CTAs per SM (two warps per scheduler), not the most the registers
    // allow: the jobs are taken longest first, and a long job that shares its
    // scheduler with others ends the launch alone.  One CTA where even beside
    // one other the longest job would outlast the launch's ideal time (every
    // scheduler busy).  Fills of both rounds on GB300, pairs of 2-20 kb, one /
    // two CTAs: 2,000 pairs 5.9 / 6.8 ms, 10,000 pairs 11.4 / 12.2 ms, 20,000
    // pairs 22.7 / 20.3 ms.  NW_BBAND_OCC overrides (sweeps).
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
        wt[q] = BitsWalkTask{it.ptr_off, mpos, it.a_slot, it.b_slot, it.m, it.n, it.shape.g * it.shape.Q, it.shape.hi,
                             it.shape.a_first, (uint32_t)q};
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
    if ((rc = scratch(ctx, "bband_trace_tasks", tt.size() * sizeof(TraceTask) + 16, &v))) return rc;
    TraceTask *dtt = (TraceTask *)v;
    cudaError_t e = cudaMemcpyAsync(dw, wt.data(), wt.size() * sizeof(BitsWalkTask), cudaMemcpyHostToDevice,
                                    ctx->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dtt, tt.data(), tt.size() * sizeof(TraceTask), cudaMemcpyHostToDevice, ctx->stream);
    // the host task arrays go out of scope: wait for their copies (the fill
    // before them has finished already; its scores were read back), not for
    // the walk, so the caller prepares its next round while the GPU walks
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "walk tasks H2D");
    {
        LaunchTimer t(ctx, "bband_walk");
        // one warp per CTA; its 48 KB of records let four CTAs share an SM (one warp per scheduler)
        constexpr int smem = kSubPairs * kBlockSteps * kSubWords * (int)sizeof(uint4);
        static_assert(smem <= 48 * 1024, "above the default limit of dynamic shared memory");
        const uint32_t blocks = (uint32_t)std::min<size_t>((which.size() + kSubPairs - 1) / kSubPairs, 65535);
        const BitsWalkArgs wa{planes.pl0, planes.pl1, planes.max_base, (const uint4 *)ptr, dw, (uint32_t)which.size(),
                              (uint8_t *)mv, (uint64_t *)nm, ctx->d_err};
        k_bits_walk<<<blocks, 32, smem, ctx->stream>>>(wa);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(ctx, e, "walk launch");
    return launch_finish(ctx, TraceTask{}, dtt, (uint32_t)tt.size(), mflag);
}

}  // namespace nw
