// Bit-sliced score-only fill (a3/a7): the Sec. 2.3 recurrence from the
// Sec. 2.2 boundary, 32 cells per machine word.
//
// Difference form.  In the W domain (W = H - gap*(i+j), see nw_internal.cuh)
// gaps cost nothing and a diagonal step gains s' = s - 2*gap, so W never
// decreases along a row or a column and never gains more than s'max over its
// diagonal neighbour.  With
//     dH(i,j) = W(i,j) - W(i,j-1),   dV(i,j) = W(i,j) - W(i-1,j),
// both lie in [0, s'max], and the recurrence becomes, for a = dH(i-1,j) (the
// cell above, against its left neighbour) and b = dV(i,j-1) (the cell to the
// left, against its upper neighbour):
//     T = W(i,j) - W(i-1,j-1) = max(s'(i,j), a, b),
//     dV(i,j) = T - a,   dH(i,j) = T - b.
// When 0 <= s'(mismatch) <= s'(match) <= 3 -- the paper's +1/-1/-1 gives 3
// and 1 -- every value fits in two bits, and a 32-bit word holds one bit of
// 32 cells: a "plane".  A lane keeps the planes of 32 consecutive rows on one
// anti-diagonal (bit p = row top + p); the cell above a bit is the bit below
// it on the previous anti-diagonal and the cell to its left is the same bit,
// so one anti-diagonal step is a fixed sequence of funnel shifts and
// three-input logic operations (LOP3) on whole words.
//
// Work split.  One pair per lane.  A lane holds K = 1, 2 or 4 words of each
// plane, rows dealt out in turn: bit p of word w is row K*p + w of a stripe of
// 32*K rows.  So the cell above word w is the same bit of word w - 1 one step
// earlier -- no shift --, only word 0 takes a funnel shift of word K - 1; and
// the B window of word w is the one word 0 had w steps before, so K windows
// are kept, and each step one of them moves by one bit.  The shifts (the
// upper dH, the stripe boundary and the B window, two planes each) cost a step
// 6 operations for all K words, the cells 10 a word: 16, 13 or 11.5 a word.
//
// Stripes are aligned to the bottom of the grid (the last row of the last
// stripe is row m) and follow one another without a gap: the row r of a
// stripe starts r steps after its row 0, on a period of whole chunks of 32
// columns, so while the last rows finish a stripe the first ones are in the
// next.  A step starts one row: its bit of A is replaced and its dV cleared.
// The rows <= 0 of the first stripe are padding: what they hold is kept from
// row 1 by a mask on its upper dH.  The previous stripe's bottom row arrives
// as 32 input bits per chunk and the stripe's own leaves through the same
// shift register; the words go through a per-warp buffer in global memory,
// [chunk][lane], so a warp's accesses coalesce.  The lanes of a warp hold
// pairs of equal stripe count and similar width (a "job"), so they run in
// lockstep; jobs are taken longest first from an atomic counter.  The score is
// W(m,n) = sum over j of dH(m,j), read from the last stripe's outgoing words
// with population counts.
//
// What bounds it: the logic pipe.  All-vs-all of 512 sequences of 500 to
// 1,500 bases: 3.2 ms; with one word a lane and a gap of 31 steps after each
// stripe 4.2 ms.  (K = 1, 2, 4 for all: 4.3, 3.4, 3.25 ms; 20,000 pairs of
// reads of 50 to 600 bases .43, .36, .34 ms.)
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <vector>

#include "nw_bits.cuh"
#include "nw_bits_shape.h"
#include "nw_order.h"

namespace nw {

// The cell update for any scoring of two bit planes (see bits_cell).
__device__ __forceinline__ void bits_cell_gen(const BitsScoring &g, uint32_t eq, uint32_t a0, uint32_t a1, uint32_t b0,
                                              uint32_t b1, uint32_t &H0, uint32_t &H1, uint32_t &V0, uint32_t &V1) {
    const uint32_t p = lop3<kLutAndOrNot>(a0, a1, b1);  // the low bit of max(a, b), from a
    const uint32_t q = lop3<kLutAndOrNot>(b0, b1, a1);  // ... from b
    const uint32_t e1 = lop3<kLutSel>(eq, g.M1, g.X1), e0 = lop3<kLutSel>(eq, g.M0, g.X0);
    const uint32_t m0 = p | q, m1 = a1 | b1;
    const uint32_t T0 = lop3<kLutAndNotOr>(m0, e1, m1) | lop3<kLutAndNotOr>(e0, m1, e1);
    const uint32_t T1 = m1 | e1;
    const uint32_t ca = lop3<kLutAndNot>(a0, T0, 0u), cb = lop3<kLutAndNot>(b0, T0, 0u);  // borrows
    V0 = T0 ^ a0;
    V1 = lop3<kLutXor3>(T1, a1, ca);
    H0 = T0 ^ b0;
    H1 = lop3<kLutXor3>(T1, b1, cb);
}

// A lane's state: difference planes, row bases and B windows of K words, the
// next stripe's row bases, and the mask that clears row 1's upper dH.
template <int K>
struct BitsLane {
    uint32_t H0[K], H1[K], V0[K], V1[K], A0[K], A1[K], N0[K], N1[K], B0[K], B1[K], top[K];
};

// 32 steps.  X: the chunk's columns, the first at bit 31; Q: the shift register
// of the stripe boundary (bit 31 = the input bit of the step, the output bit
// enters at bit 0).  TRANS: rows of a stripe start, one a step, from bit `q` on.
// FIRST: rows of the first stripe are at work; `lift`: the rows that start are
// beyond them.
template <bool GEN, int K, bool FIRST, bool TRANS>
__device__ __forceinline__ void bits_chunk(BitsLane<K> &s, uint32_t X0, uint32_t X1, uint32_t &Q0, uint32_t &Q1,
                                           uint32_t q, uint32_t lift, const BitsScoring &g) {
    uint32_t tb = 1u << q;
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            constexpr auto mod = [](int x) { return (x + 4) % K; };
            const int w0 = mod(u);
            s.B0[w0] = __funnelshift_l(u ? mul(X0, 1u << u) : X0, s.B0[w0], 1);
            s.B1[w0] = __funnelshift_l(u ? mul(X1, 1u << u) : X1, s.B1[w0], 1);
            if constexpr (TRANS) {
                const uint32_t bit = u / K ? mul(tb, 1u << (u / K)) : tb;
                s.A0[w0] = lop3<kLutSel>(bit, s.N0[w0], s.A0[w0]);
                s.A1[w0] = lop3<kLutSel>(bit, s.N1[w0], s.A1[w0]);
                s.V0[w0] &= ~bit;
                s.V1[w0] &= ~bit;
                if constexpr (FIRST) s.top[w0] |= bit & lift;
            }
            uint32_t a0 = __funnelshift_l(Q0, s.H0[K - 1], 1), a1 = __funnelshift_l(Q1, s.H1[K - 1], 1);
            const uint32_t h0 = a0, h1 = a1;
#pragma unroll
            for (int w = K - 1; w >= 0; --w) {
                a0 = w ? s.H0[w ? w - 1 : 0] : h0;
                a1 = w ? s.H1[w ? w - 1 : 0] : h1;
                if constexpr (FIRST) {
                    a0 &= s.top[w];
                    a1 &= s.top[w];
                }
                const uint32_t eq = lop3<kLutEq>(s.A0[w], s.B0[mod(u - w)], s.A1[w] ^ s.B1[mod(u - w)]);  // A_i == B_j
                if constexpr (GEN) bits_cell_gen(g, eq, a0, a1, s.V0[w], s.V1[w], s.H0[w], s.H1[w], s.V0[w], s.V1[w]);
                else bits_cell(eq, a0, a1, s.V0[w], s.V1[w], s.H0[w], s.H1[w], s.V0[w], s.V1[w]);
            }
            Q0 = __funnelshift_l(s.H0[K - 1], Q0, 1);
            Q1 = __funnelshift_l(s.H1[K - 1], Q1, 1);
        }
        X0 = mul(X0, 16u);
        X1 = mul(X1, 16u);
        if constexpr (TRANS) tb <<= 4 / K;
    }
}

__device__ __forceinline__ uint32_t even_bits32(uint32_t x) {  // into the low 16 bits
    x &= 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0F0F0F0Fu;
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return (x | (x >> 8)) & 0x0000FFFFu;
}

// 32*K rows from row `row` on (before the first base: unspecified), dealt out in turn to K words.
template <int K>
__device__ __forceinline__ void deal_rows(const uint32_t *pl, int64_t Ag, int32_t row, uint32_t (&out)[K]) {
    uint32_t c[K];
#pragma unroll
    for (int j = 0; j < K; ++j) c[j] = plane_window(pl, Ag + max(row + 32 * j, -32));
    if constexpr (K == 1) {
        out[0] = c[0];
    } else if constexpr (K == 2) {
        out[0] = even_bits32(c[0]) | even_bits32(c[1]) << 16;
        out[1] = even_bits32(c[0] >> 1) | even_bits32(c[1] >> 1) << 16;
    } else {
        static_assert(K == 4);
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            const uint32_t lo = even_bits32(c[0] >> o) | even_bits32(c[1] >> o) << 16;
            const uint32_t hi = even_bits32(c[2] >> o) | even_bits32(c[3] >> o) << 16;
            out[o] = even_bits32(lo) | even_bits32(hi) << 16;
            out[o + 2] = even_bits32(lo >> 1) | even_bits32(hi >> 1) << 16;
        }
    }
}

// W(m, n) of a lane's pair, in the steps of its job: job.T chunks, a stripe
// every job.C.  (Count: 64 bits only where T needs them, they cost a lone warp 3%
// of its time.)
template <bool GEN, int K, class Count = uint32_t>
__device__ __forceinline__ int32_t bits_pairs_of(const BitsArgs &p, const BitsJob &job, uint32_t m, uint32_t n,
                                                 int64_t Ag, int64_t Bg, uint2 *rows) {
    constexpr int32_t SH = 32 * K;
    const uint32_t S = job.S, C = job.C;
    const int32_t pad = SH * (int32_t)S - (int32_t)m;  // rows above row 1 in stripe 0
    const int32_t ncol = (int32_t)((n + 31) / 32);     // chunks that hold columns of this pair
    BitsLane<K> s;
#pragma unroll
    for (int w = 0; w < K; ++w) {
        s.H0[w] = s.H1[w] = s.V0[w] = s.V1[w] = s.A0[w] = s.A1[w] = s.N0[w] = s.N1[w] = s.B0[w] = s.B1[w] = 0;
        s.top[w] = pad % K == w ? ~(1u << (pad / K)) : ~0u;
    }
    const auto cols = [&](const uint32_t *pl, uint32_t cl) {
        return __brev(plane_window(pl, Bg + 32 * (int64_t)min((int32_t)cl, ncol)));
    };
    uint32_t X0 = cols(p.pl0, 0), X1 = cols(p.pl1, 0);
    uint2 prev = make_uint2(0u, 0u), nx = make_uint2(0u, 0u);
    int32_t W = 0;
    uint32_t stripe = 0, cl = 0;   // of the stripe's row 0
    uint32_t started = 0, lift = 0;  // chunks since a stripe began; all ones once it is not the first
    const Count last = bits_last_row<Count>(S, C, K), T = (Count)job.T;
    for (Count c = 0; c < T; ++c) {
        if (cl == 0 && stripe < S) {
            started = 0;
            lift = stripe ? ~0u : 0u;
            const int32_t row = SH * (int32_t)stripe - pad;
            deal_rows<K>(p.pl0, Ag, row, s.N0);
            deal_rows<K>(p.pl1, Ag, row, s.N1);
        }
        const uint32_t cn = cl + 1 == C ? 0u : cl + 1;
        const uint32_t Y0 = cols(p.pl0, cn), Y1 = cols(p.pl1, cn);  // the next chunk's columns
        // The bottom row of the stripe above: its column 32x is bit 0 of the
        // word of chunk x + K - 1, the 31 columns that follow are the high bits
        // of the word after it.  Loaded one chunk ahead; the buffer holds the
        // last C chunks' words.
        uint32_t Q0 = 0, Q1 = 0;
        if (stripe) {
            Q0 = __funnelshift_r(nx.x, prev.x, 1);
            Q1 = __funnelshift_r(nx.y, prev.y, 1);
        }
        prev = nx;
        if (S > 1 && c + 2 >= C) {
            uint32_t r = cl + 1 + K;
            if (r >= C) r -= C;
            nx = __ldcg(rows + (size_t)r * 32u);
        }
        if (c < C + K || S == 1) {
            if (started < (uint32_t)K) bits_chunk<GEN, K, true, true>(s, X0, X1, Q0, Q1, started * (32 / K), lift, p.g);
            else bits_chunk<GEN, K, true, false>(s, X0, X1, Q0, Q1, 0u, 0u, p.g);
        } else {
            if (started < (uint32_t)K) bits_chunk<GEN, K, false, true>(s, X0, X1, Q0, Q1, started * (32 / K), 0u, p.g);
            else bits_chunk<GEN, K, false, false>(s, X0, X1, Q0, Q1, 0u, 0u, p.g);
        }
        ++started;
        // outgoing bits: bit b is column 32 (c - K + 1) - b of the bottom row, from the stripe's first chunk on
        if (S > 1 && c <= last) __stcg(rows + (size_t)cl * 32u, make_uint2(Q0, Q1));
        int32_t lo, hi;
        bits_last_row_span((uint32_t)(c - last), n, lo, hi);
        if (c >= last && lo <= hi) {
            const uint32_t mk = (hi == 31 ? ~0u : ((2u << hi) - 1u)) & (~0u << lo);
            W += __popc(Q0 & mk) + 2 * __popc(Q1 & mk);
        }
        X0 = Y0;
        X1 = Y1;
        cl = cn;
        if (cl == 0) ++stripe;
    }
    return W;
}

// Row and column of the q-th pair of a class: the columns before the class's
// rows pair with all of them, a column among them with the rows after it.
__device__ __forceinline__ void class_pair(const BitsClass &k, uint32_t q, uint32_t &r, uint32_t &c) {
    const uint32_t rows = k.r1 - k.r0, whole = k.r0 * rows;
    if (q < whole) {
        c = q / rows;
        r = k.r0 + q % rows;
        return;
    }
    // the x-th column among the rows starts at x (2 rows - x - 1) / 2
    const uint64_t t = q - whole, b = 2ull * rows - 1ull;
    uint64_t x = (uint64_t)(((double)b - sqrt(fmax((double)(b * b) - 8.0 * (double)t, 0.0))) * 0.5);
    if (x > rows - 2ull) x = rows - 2ull;
    while (x > 0 && x * (b - x) / 2ull > t) --x;
    while ((x + 1ull) * (b - x - 1ull) / 2ull <= t) ++x;
    c = k.r0 + (uint32_t)x;
    r = c + 1u + (uint32_t)(t - x * (b - x) / 2ull);
}

// The warps of a launch take its jobs.  WIDE: jobs of 2^32 chunks or more.
template <bool GEN, bool WIDE>
__device__ __forceinline__ void bits_jobs(const BitsArgs &p) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    uint2 *rows = p.rows + (size_t)gw * p.rows_chunks * 32u + lane;
    for (;;) {
        uint32_t jid = 0;
        if (lane == 0) jid = atomicAdd(p.counter, 1u);
        jid = __shfl_sync(kFull, jid, 0);
        if (jid >= p.njobs) break;
        const BitsJob job = p.jobs[jid];
        const bool active = lane < job.cnt;
        uint32_t m, n, aw, bw, out0, out1;
        if (p.tasks) {
            const BitsTask tk = p.tasks[job.t0 + (active ? lane : 0u)];
            m = tk.m;
            n = tk.n;
            aw = tk.aw;
            bw = tk.bw;
            out0 = tk.out0;
            out1 = tk.out1;
        } else {
            uint32_t r, c;
            class_pair(p.classes[job.cls], job.t0 + (active ? lane : 0u), r, c);
            const BitsSeq a = p.seqs[r], b = p.seqs[c];
            m = a.len;
            n = b.len;
            aw = a.w;
            bw = b.w;
            out0 = a.id * p.nseq + b.id;
            out1 = b.id * p.nseq + a.id;
        }
        int32_t W = 0;
        const int64_t Ag = (int64_t)aw * 32 - kPlanePad, Bg = (int64_t)bw * 32 - kPlanePad;  // planar slots
        if (job.S) {
            if constexpr (WIDE) W = bits_pairs_of<GEN, 1, uint64_t>(p, job, m, n, Ag, Bg, rows);
            else if (job.K == 4) W = bits_pairs_of<GEN, 4>(p, job, m, n, Ag, Bg, rows);
            else if (job.K == 2) W = bits_pairs_of<GEN, 2>(p, job, m, n, Ag, Bg, rows);
            else W = bits_pairs_of<GEN, 1>(p, job, m, n, Ag, Bg, rows);
        }
        if (active) {
            const int32_t sc = W * p.unit + p.gap * (int32_t)(m + n);
            if (in_range(out0, p.score_cap, p.err, kSiteBatchScore)) p.scores[out0] = sc;
            if (out1 != ~0u && in_range(out1, p.score_cap, p.err, kSiteBatchScore)) p.scores[out1] = sc;
        }
    }
}

template <bool GEN>
__global__ void __launch_bounds__(kBitsWarps * 32) k_bits_score(BitsArgs p) {
    bits_jobs<GEN, false>(p);
}
// (a kernel of its own: the second count in the first one's code cost a lone warp 5%)
template <bool GEN>
__global__ void __launch_bounds__(kBitsWarps * 32) k_bits_wide(BitsArgs p) {
    bits_jobs<GEN, true>(p);
}

// Planar copy of a sequence by a warp: word w of its slot holds bit k of the
// codes of its bases 32w .. 32w+31 (bases past its end read as 0).
__device__ __forceinline__ void plane_copy(const uint8_t *src, uint32_t nbytes, uint32_t dst, uint32_t lane,
                                           uint32_t *pl0, uint32_t *pl1) {
    const uint32_t words = (nbytes + 7) / 8;
    for (uint32_t w = lane; w < words; w += 32) {
        uint64_t v = 0;
        const uint32_t b0 = 8 * w;
        if (b0 + 8 <= nbytes) {
#pragma unroll
            for (int k = 0; k < 8; ++k) v |= (uint64_t)src[b0 + k] << (8 * k);
        } else {
            for (uint32_t k = 0; b0 + k < nbytes; ++k) v |= (uint64_t)src[b0 + k] << (8 * k);
        }
        pl0[dst + w] = even_bits(v);
        pl1[dst + w] = even_bits(v >> 1);
    }
}

// The launch's distinct sequences, one warp per sequence.
__global__ void k_planes(const uint8_t *pool, const PlaneSeg *segs, uint32_t nsegs, uint32_t *pl0, uint32_t *pl1) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t sg = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; sg < nsegs; sg += (gridDim.x * blockDim.x) >> 5) {
        const PlaneSeg seg = segs[sg];
        const uint8_t *src = pool ? pool + seg.src : reinterpret_cast<const uint8_t *>(seg.src);  // offset or address
        plane_copy(src, seg.nbytes, seg.dst, lane, pl0, pl1);
    }
}

// Both sequences of every task, into the task's own slots.
__global__ void k_planes_tasks(const uint8_t *pool, const BitsTask *tasks, uint32_t ntasks, uint32_t *pl0,
                               uint32_t *pl1) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < 2 * ntasks;
         k += (gridDim.x * blockDim.x) >> 5) {
        const BitsTask t = tasks[k >> 1];
        if (!t.m || !t.n) continue;  // no slots
        if (k & 1u) plane_copy(pool + t.b_off, (t.n + 3) / 4, t.bw, lane, pl0, pl1);
        else plane_copy(pool + t.a_off, (t.m + 3) / 4, t.aw, lane, pl0, pl1);
    }
}

// ------------------------------------------------------------------ host
static size_t plane_hash(uint64_t off, uint32_t len) {
    uint64_t z = off * 0x9E3779B97F4A7C15ull ^ ((uint64_t)len << 17);
    z ^= z >> 31;
    z *= 0xBF58476D1CE4E5B9ull;
    return (size_t)(z ^ (z >> 29));
}

void PlaneSet::rehash(size_t size) {
    std::vector<Entry> old;
    old.swap(table_);
    table_.assign(size, Entry{0, 0, 0, 0});
    for (const Entry &e : old) {
        if (!e.used) continue;
        size_t h = plane_hash(e.off, e.len) & (size - 1);
        while (table_[h].used) h = (h + 1) & (size - 1);
        table_[h] = e;
    }
}

void PlaneSet::reserve(size_t n) {
    size_t size = 64;
    while (size < 2 * n) size *= 2;
    if (size > table_.size()) rehash(size);
    segs_.reserve(n);
}

int64_t PlaneSet::add(uint64_t off, uint32_t len) {
    if (2 * (count_ + 1) > table_.size()) rehash(std::max<size_t>(64, 2 * table_.size()));
    const size_t mask = table_.size() - 1;
    size_t h = plane_hash(off, len) & mask;
    for (; table_[h].used; h = (h + 1) & mask)
        if (table_[h].off == off && table_[h].len == len) return table_[h].slot;
    const uint32_t nbytes = (len + 3) / 4;
    const int64_t slot = (int64_t)words_ * 32 - kPlanePad;
    segs_.push_back(PlaneSeg{off, nbytes, (uint32_t)words_});
    words_ += (nbytes + 7) / 8 + 2;
    table_[h] = Entry{off, len, 1, slot};
    ++count_;
    return slot;
}

int PlaneSet::prepare(nw_ctx *ctx, const std::string &prefix) {
    int rc;
    void *v = nullptr;
    const uint64_t words = words_ + 4;  // room for the last window's second word
    if (words >= (1ull << 32)) return fail(ctx, NW_ERR_ARG, "planar copy of more than 2^37 bases");
    if ((rc = scratch(ctx, (prefix + "_planes").c_str(), (size_t)words * 8, &v))) return rc;
    planes_ = (uint32_t *)v;
    pl0 = planes_;
    pl1 = planes_ + words;
    max_base = (int64_t)words * 32 - kPlanePad - 64;
    if ((rc = scratch(ctx, (prefix + "_plane_segs").c_str(), segs_.size() * sizeof(PlaneSeg) + 16, &v))) return rc;
    dsegs_ = (PlaneSeg *)v;
    if (!segs_.empty()) {
        cudaError_t e = cudaMemcpyAsync(dsegs_, segs_.data(), segs_.size() * sizeof(PlaneSeg), cudaMemcpyHostToDevice,
                                        ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);  // the table is host memory of this object
        if (e != cudaSuccess) return cuda_fail(ctx, e, "planar segments H2D");
    }
    return NW_OK;
}

int PlaneSet::enqueue(nw_ctx *ctx, const uint8_t *pool) const {
    if (segs_.empty()) return NW_OK;
    {
        LaunchTimer t(ctx, "planes");
        const uint32_t blocks = (uint32_t)std::min<size_t>((segs_.size() + 7) / 8, 4096);
        k_planes<<<blocks, 256, 0, ctx->stream>>>(pool, dsegs_, (uint32_t)segs_.size(), planes_,
                                                  planes_ + (words_ + 4));
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "planar copy launch");
}

int PlaneSet::launch(nw_ctx *ctx, const uint8_t *pool, const std::string &prefix) {
    const int rc = prepare(ctx, prefix);
    return rc ? rc : enqueue(ctx, pool);
}

BitsUnits bits_units(const nw_scoring &sc) {
    const int32_t sm = sc.match - 2 * sc.gap, sx = sc.mismatch - 2 * sc.gap;
    const int32_t unit = sm > 0 && sx >= 0 ? std::gcd(sm, sx) : 1;
    return BitsUnits{sm / unit, sx / unit, unit};
}

bool bits_scoring_ok(const nw_scoring &sc) {
    const int32_t sm = sc.match - 2 * sc.gap, sx = sc.mismatch - 2 * sc.gap;
    return sx >= 0 && sx <= sm && sm <= 3;
}

bool bits_batch_ok(const nw_scoring &sc) {
    const BitsUnits u = bits_units(sc);
    return u.sx >= 0 && u.sx <= u.sm && u.sm <= 3;
}

// The K with the least work at as many columns as rows, by the rows' words (a
// pair's columns are mostly as many or more): more words take fewer shifts a
// word, but pad the rows to 32*K and want a period of K + 3 chunks for the row
// buffer (a word is read K + 1 chunks after its stripe's first, one chunk
// ahead of its use).  From 64 words on the padding no longer matters.
// NW_BITS_WORDS: one K for all (sweeps).
class BitsShapes {
  public:
    BitsShapes() {
        const char *e = getenv("NW_BITS_WORDS");
        const uint32_t force = e ? (uint32_t)atoi(e) : 0u;
        for (uint32_t w = 1; w <= kWords; ++w) {
            uint64_t best = ~0ull;
            for (uint32_t l = 0; l < 3; ++l) {
                const BitsShape c = shape(w, l);
                const uint64_t x = force ? (force != c.K) : c.work(32 * w);
                if (x < best) {
                    best = x;
                    by_words_[w] = c;
                }
            }
        }
    }
    // m = 0: no stripes.  Rows that with n columns come to 2^32 chunks or more run
    // one word a lane, the form that counts in 64 bits.
    BitsShape of(uint32_t m, uint32_t n) const {
        const uint32_t w = (m + 31) / 32;
        if (w <= kWords) return by_words_[w];
        const BitsShape s = shape(w, by_words_[kWords].K / 2);
        return s.chunks(n) >> 32 ? shape(w, 0) : s;
    }

  private:
    static constexpr uint32_t kWords = 64;
    // K = 2^l
    static BitsShape shape(uint32_t w, uint32_t l) { return BitsShape{1u << l, (w + (1u << l) - 1) >> l, (10u << l) + 6}; }
    BitsShape by_words_[kWords + 1] = {};
};

// A job of pairs of at most n columns.
static BitsJob job_of(const BitsShape &s, uint32_t n, uint32_t t0, uint32_t cnt, uint32_t cls) {
    return BitsJob{s.S ? s.chunks(n) : 0u, t0, cnt, s.S, s.S ? s.period(n) : 0u, s.K, cls};
}

// The launch's tables in one upload, its constants, grid and row buffers.
// `head`: the task table, or the sequence and class tables (16-byte padded).
static int bits_finish_plan(nw_ctx *ctx, const uint8_t *pool, std::vector<uint8_t> &head, std::vector<BitsJob> &jobs,
                            uint32_t maxC, const nw_scoring &sc, int32_t *scores, uint32_t score_cap,
                            const std::string &prefix, BitsPlan *plan, void **dhead) {
    int rc;
    // longest jobs first, ties in job order
    std::vector<uint64_t> keys(jobs.size());
    uint64_t most = 0;
    for (size_t q = 0; q < jobs.size(); ++q) {
        keys[q] = jobs[q].T * (10 * jobs[q].K + 6);
        most = std::max(most, jobs[q].T);
    }
    std::vector<uint32_t> jo = radix_order_desc(std::move(keys));
    // jobs of 2^32 chunks or more lead: they have a launch of their own
    plan->wide = 0;
    if (most >> 32)
        plan->wide = (uint32_t)(std::stable_partition(jo.begin(), jo.end(), [&](uint32_t q) { return jobs[q].T >> 32; }) - jo.begin());
    const size_t jobs_at = (head.size() + 15) / 16 * 16;
    head.resize(jobs_at + jobs.size() * sizeof(BitsJob));
    BitsJob *hj = reinterpret_cast<BitsJob *>(head.data() + jobs_at);
    for (size_t q = 0; q < jobs.size(); ++q) hj[q] = jobs[jo[q]];
    if ((rc = plan->planes.prepare(ctx, prefix))) return rc;
    BitsArgs &ba = plan->ba;
    ba.pl0 = plan->planes.pl0;
    ba.pl1 = plan->planes.pl1;
    void *v = nullptr;
    if ((rc = scratch(ctx, (prefix + "_bits_plan").c_str(), head.size() + 16, &v))) return rc;
    cudaError_t e = cudaMemcpyAsync(v, head.data(), head.size(), cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);  // the host table is temporary
    if (e != cudaSuccess) return cuda_fail(ctx, e, "bit-sliced plan upload");
    *dhead = v;
    ba.jobs = reinterpret_cast<const BitsJob *>((const uint8_t *)v + jobs_at);
    ba.njobs = (uint32_t)jobs.size();
    ba.scores = scores;
    ba.score_cap = score_cap;
    ba.gap = sc.gap;
    ba.err = ctx->d_err;
    const BitsUnits u = bits_units(sc);
    ba.unit = u.unit;
    ba.g = u.planes();
    plan->gen = u.gen();
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, plan->gen ? k_bits_score<true> : k_bits_score<false>,
                                                  kBitsWarps * 32, 0);
    // One CTA of 8 warps per SM (two warps per scheduler), not the most the
    // registers allow: with more, the longest jobs -- taken first -- share
    // their scheduler with the rest and finish the launch alone.  All-vs-all of
    // 512 sequences: 3.25 ms, with two CTAs 3.6.  NW_BITS_OCC overrides (sweeps).
    int cap = 1;
    if (const char *e = getenv("NW_BITS_OCC")) cap = std::max(1, atoi(e));
    occ = std::min(occ, cap);
    if (occ < 1) occ = 1;
    uint32_t blocks = (uint32_t)occ * (uint32_t)ctx->sm_count;
    const uint32_t need = (ba.njobs + kBitsWarps - 1) / kBitsWarps;
    plan->blocks = std::max(1u, std::min(blocks, need));
    ba.rows_chunks = maxC;
    if ((rc = scratch(ctx, (prefix + "_bits_rows").c_str(),
                      (size_t)plan->blocks * kBitsWarps * maxC * 32 * sizeof(uint2), &v)))
        return rc;
    ba.rows = (uint2 *)v;
    if ((rc = scratch(ctx, (prefix + "_bits_counter").c_str(), 16, &v))) return rc;
    ba.counter = (uint32_t *)v;
    plan->pool = pool;
    return NW_OK;
}

// bits_prepare with the distinct sequences' slots (`shared`) or with one for each
// of a task's sequences where that is the cheaper plan; *own: which it took.
static int bits_prepare_slots(nw_ctx *ctx, const uint8_t *pool, const std::vector<BatchTask> &tasks, const nw_scoring &sc,
                              int32_t *scores, uint32_t score_cap, const std::string &prefix, BitsPlan *plan, bool shared,
                              bool *own_out) {
    *plan = BitsPlan{};
    HostTimer ht(ctx, "bits_plan");
    // rows: the orientation with less work (the score is symmetric); order:
    // equal shapes, widest first
    const BitsShapes shapes;
    const size_t n = tasks.size();
    std::vector<uint64_t> keys(n);
    std::vector<uint8_t> turned(n);
    uint64_t bytes = 0, extent = 0;
    for (size_t k = 0; k < n; ++k) {
        const BatchTask &t = tasks[k];
        if (!t.m || !t.n) {
            keys[k] = std::max(t.m, t.n);  // no stripes
            continue;
        }
        BitsShape sh = shapes.of(t.m, t.n);
        if ((t.m + 31) / 32 != (t.n + 31) / 32) {
            const BitsShape sn = shapes.of(t.n, t.m);
            turned[k] = sn.work(t.m) < sh.work(t.n);
            if (turned[k]) sh = sn;
        }
        keys[k] = (uint64_t)sh.S << 36 | (uint64_t)sh.K << 32 | (turned[k] ? t.m : t.n);
        bytes += (t.m + 3) / 4 + (t.n + 3) / 4;
        extent = std::max(extent, std::max(t.a_off + (t.m + 3) / 4, t.b_off + (t.n + 3) / 4));
    }
    const std::vector<uint32_t> order = radix_order_desc(std::move(keys));
    // Planar copies: a slot for each of a task's sequences, unless the tasks
    // read their sequences several times over (then the distinct sequences,
    // found by hashing, which costs the host more than the device saves
    // otherwise: 20,000 pairs of distinct reads, 1 ms) -- or may do so, when
    // the slots (as many bytes as the packed bases, and at most 24 more a
    // sequence) would take more than a quarter of the scratch that is left: few
    // sequences far up in a large pool.
    const uint64_t slots = bytes + 48 * (uint64_t)n;
    const bool own = !shared && bytes <= 2 * extent && slots < (1ull << 35) &&
                     slots <= scratch_headroom(ctx, (prefix + "_planes").c_str()) / 4;
    *own_out = own;
    uint64_t words = 2;
    if (!own) plan->planes.reserve(std::min<size_t>(2 * n, 1u << 16));
    std::vector<uint8_t> head(n * sizeof(BitsTask));
    BitsTask *ht_ = reinterpret_cast<BitsTask *>(head.data());
    std::vector<BitsJob> jobs;
    uint32_t maxC = 1;
    for (size_t q = 0; q < n; ++q) {
        const BatchTask &t = tasks[order[q]];
        BitsTask b{t.a_off, t.b_off, 2, 2, t.m, t.n, t.out0, t.out1};
        if (turned[order[q]]) {
            std::swap(b.a_off, b.b_off);
            std::swap(b.m, b.n);
        }
        const BitsShape sh = shapes.of(b.n ? b.m : 0, b.n);
        if (sh.S && own) {
            b.aw = (uint32_t)words;
            b.bw = b.aw + (b.m + 31) / 32 + 2;
            words = (uint64_t)b.bw + (b.n + 31) / 32 + 2;
        } else if (sh.S) {
            b.aw = PlaneSet::word_of(plan->planes.add(b.a_off, b.m));
            b.bw = PlaneSet::word_of(plan->planes.add(b.b_off, b.n));
        }
        ht_[q] = b;
        if (jobs.empty() || jobs.back().S != sh.S || jobs.back().K != sh.K || jobs.back().cnt == 32)
            jobs.push_back(job_of(sh, b.n, (uint32_t)q, 0, 0));
        ++jobs.back().cnt;
        maxC = std::max(maxC, jobs.back().C);
    }
    if (own) {
        plan->planes.reserve_words(words - 2);
        plan->ntasks = (uint32_t)n;
    }
    void *dh = nullptr;
    const int rc = bits_finish_plan(ctx, pool, head, jobs, maxC, sc, scores, score_cap, prefix, plan, &dh);
    plan->ba.tasks = (const BitsTask *)dh;
    return rc;
}

void bits_release(nw_ctx *ctx, const std::string &prefix) {
    free_prefix(ctx, prefix + "_plane");
    free_prefix(ctx, prefix + "_bits");
}

int bits_prepare(nw_ctx *ctx, const uint8_t *pool, const std::vector<BatchTask> &tasks, const nw_scoring &sc,
                 int32_t *scores, uint32_t score_cap, const std::string &prefix, BitsPlan *plan) {
    *plan = BitsPlan{};
    if (tasks.empty()) return NW_OK;
    const std::string before = ctx->msg;
    bool own = false;
    int rc = bits_prepare_slots(ctx, pool, tasks, sc, scores, score_cap, prefix, plan, false, &own);
    if (rc == NW_ERR_OOM && own) {  // the sequences' own slots left too little for the rest
        bits_release(ctx, prefix);
        ctx->msg = before;
        rc = bits_prepare_slots(ctx, pool, tasks, sc, scores, score_cap, prefix, plan, true, &own);
    }
    return rc;
}

int bits_prepare_all(nw_ctx *ctx, const uint8_t *pool, const uint64_t *off, const uint32_t *len, uint32_t nseq,
                     const nw_scoring &sc, int32_t *scores, const std::string &prefix, BitsPlan *plan) {
    *plan = BitsPlan{};
    HostTimer ht(ctx, "bits_plan");
    std::vector<uint64_t> keys(nseq);
    for (uint32_t i = 0; i < nseq; ++i) keys[i] = len[i];
    const std::vector<uint32_t> order = radix_order_desc(std::move(keys));
    plan->planes.reserve(nseq);
    const size_t classes_at = (nseq * sizeof(BitsSeq) + 15) / 16 * 16;
    std::vector<BitsSeq> seqs(nseq);
    for (uint32_t q = 0; q < nseq; ++q) {
        const uint32_t i = order[q];
        seqs[q] = BitsSeq{len[i] ? PlaneSet::word_of(plan->planes.add(off[i], len[i])) : 2u, len[i], i};
    }
    const BitsShapes shapes;
    std::vector<BitsClass> classes;
    std::vector<BitsJob> jobs;
    jobs.reserve((uint64_t)nseq * nseq / 64 + 64);  // 32 pairs a job, and a class's last
    uint32_t maxC = 1;
    const uint32_t widest = nseq ? seqs[0].len : 0u;
    for (uint32_t r0 = 0; r0 < nseq;) {
        const BitsShape sh = shapes.of(seqs[r0].len, widest);
        uint32_t r1 = r0 + 1;
        for (; r1 < nseq; ++r1)
            if (const BitsShape x = shapes.of(seqs[r1].len, widest); x.S != sh.S || x.K != sh.K) break;
        const uint32_t rows = r1 - r0, pairs = r0 * rows + rows * (rows - 1) / 2;
        // the pairs run through the columns in order: a job's first column is its widest
        uint32_t c = ~0u, end = 0;
        BitsJob j{};
        auto end_of = [&](uint32_t col) {  // pairs of the columns up to col
            const uint32_t x = col < r0 ? 0u : col - r0 + 1u;
            return col < r0 ? (col + 1u) * rows : r0 * rows + (uint32_t)((uint64_t)x * (2ull * rows - x - 1u) / 2u);
        };
        for (uint32_t q = 0; q < pairs; q += 32) {
            if (end <= q) {
                do end = end_of(++c);
                while (end <= q);
                j = job_of(sh, seqs[c].len, 0, 0, (uint32_t)classes.size());
                maxC = std::max(maxC, j.C);
            }
            j.t0 = q;
            j.cnt = std::min(32u, pairs - q);
            jobs.push_back(j);
        }
        classes.push_back(BitsClass{r0, r1});
        r0 = r1;
    }
    std::vector<uint8_t> head(classes_at + classes.size() * sizeof(BitsClass));
    memcpy(head.data(), seqs.data(), nseq * sizeof(BitsSeq));
    memcpy(head.data() + classes_at, classes.data(), classes.size() * sizeof(BitsClass));
    void *dh = nullptr;
    const int rc = bits_finish_plan(ctx, pool, head, jobs, maxC, sc, scores, nseq * nseq, prefix, plan, &dh);
    plan->ba.seqs = (const BitsSeq *)dh;
    plan->ba.classes = (const BitsClass *)((const uint8_t *)dh + classes_at);
    plan->ba.nseq = nseq;
    return rc;
}

int bits_launch(nw_ctx *ctx, const BitsPlan &plan) {
    if (plan.ba.njobs == 0) return NW_OK;
    cudaMemsetAsync(plan.ba.counter, 0, 8, ctx->stream);
    if (plan.ntasks) {
        LaunchTimer t(ctx, "planes");
        const uint32_t blocks = std::min<uint32_t>((plan.ntasks + 3) / 4, 4096);
        k_planes_tasks<<<blocks, 256, 0, ctx->stream>>>(plan.pool, plan.ba.tasks, plan.ntasks, plan.planes.planes(),
                                                        plan.planes.planes() + plan.planes.plane_words());
    } else if (int rc = plan.planes.enqueue(ctx, plan.pool)) {
        return rc;
    }
    BitsArgs ba = plan.ba;
    if (plan.wide) {
        LaunchTimer t(ctx, "bits_wide");
        ba.njobs = plan.wide;
        ++ba.counter;
        if (plan.gen) k_bits_wide<true><<<plan.blocks, kBitsWarps * 32, 0, ctx->stream>>>(ba);
        else k_bits_wide<false><<<plan.blocks, kBitsWarps * 32, 0, ctx->stream>>>(ba);
        ba = plan.ba;
        ba.jobs += plan.wide;
        ba.njobs -= plan.wide;
    }
    if (ba.njobs) {
        LaunchTimer t(ctx, "bits_score");
        if (plan.gen) k_bits_score<true><<<plan.blocks, kBitsWarps * 32, 0, ctx->stream>>>(ba);
        else k_bits_score<false><<<plan.blocks, kBitsWarps * 32, 0, ctx->stream>>>(ba);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "bit-sliced launch");
}

}  // namespace nw
