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
// three-input logic operations (LOP3) on whole words: about 20 instructions
// for 32 cells, where the scalar kernels spend 3 per cell.
//
// Work split.  One pair per lane.  Stripes of 32 rows are aligned to the
// bottom of the grid (the last stripe's bit 31 is row m); rows <= 0 of the
// first stripe are padding, forced to the boundary's zero differences by a
// row mask.  A stripe sweeps the anti-diagonals that cross it, in chunks of
// 32 steps: bit 0 meets column t+1 at step t, bit 31 column t-30.  The
// previous stripe's bottom row arrives as 32 input bits per chunk and the
// stripe's own bottom row leaves through the same shift register (one funnel
// shift per plane and step does both); the words go through a per-warp row
// buffer in global memory, [chunk][lane], so a warp's accesses coalesce.
// The lanes of a warp hold pairs of equal stripe count and similar width
// (a "job"), so they run in lockstep; jobs are taken longest first from an
// atomic counter.  The score is W(m,n) = sum over j of dH(m,j), read from the
// last stripe's outgoing words with population counts.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <vector>

#include "nw_bits.cuh"
#include "nw_order.h"

namespace nw {

// One anti-diagonal step of the 32 cells of a lane.  (H, V): the dH, dV
// planes of the previous anti-diagonal; Q: the shift register of the stripe
// boundary (bit 31 = the input bit of this step, the output bit enters at
// bit 0).  bw: the B window (bit p = base of column t+1-p), A: the row bases,
// rmask: rows of the grid (the padding rows of a pair's first stripe, FIRST,
// keep the boundary's zero differences).  RAMP: the first chunk of a stripe,
// where bits p > u lie in column <= 0 and their dV is forced to the
// boundary's 0.
//
// What bounds it: the logic pipe, 16 operations for 32 cells (two B window
// shifts, two for equality, two to bring the upper dH into line, eight for
// the update, two for the shift register).
template <bool GEN, bool RAMP, bool FIRST>
__device__ __forceinline__ void bits_step(int u, uint32_t &H0, uint32_t &H1, uint32_t &V0, uint32_t &V1, uint32_t &Q0,
                                          uint32_t &Q1, uint32_t A0, uint32_t A1, uint32_t bw0, uint32_t bw1,
                                          uint32_t rmask, const BitsScoring &g, uint32_t X1r, uint32_t X0r) {
    const uint32_t a0 = __funnelshift_l(Q0, H0, 1), a1 = __funnelshift_l(Q1, H1, 1);  // dH of the cell above
    const uint32_t b0 = V0, b1 = V1;                                                  // dV of the cell to the left
    if constexpr (!GEN) {
        const uint32_t eq = lop3<kLutEq>(A0, bw0, A1 ^ bw1);  // A_i == B_j
        bits_cell(eq, a0, a1, b0, b1, H0, H1, V0, V1);
        if constexpr (FIRST) {
            H0 &= rmask;
            H1 &= rmask;
            V0 &= rmask;
            V1 &= rmask;
        }
        if constexpr (RAMP) {
            const uint32_t mk = (2u << u) - 1u;  // bits in column >= 1
            V0 &= mk;
            V1 &= mk;
        }
    } else {
        const uint32_t x = lop3<kLutXorOrNotC>(A1, bw1, rmask);
        const uint32_t eq = lop3<kLutEq>(A0, bw0, x);  // A_i == B_j (0 on padding rows)
        const uint32_t p = lop3<kLutAndOrNot>(a0, a1, b1);  // the low bit of max(a, b), from a
        const uint32_t q = lop3<kLutAndOrNot>(b0, b1, a1);  // ... from b
        const uint32_t e1 = lop3<kLutSel>(eq, g.M1, X1r), e0 = lop3<kLutSel>(eq, g.M0, X0r);
        const uint32_t m0 = p | q, m1 = a1 | b1;
        const uint32_t T0 = lop3<kLutAndNotOr>(m0, e1, m1) | lop3<kLutAndNotOr>(e0, m1, e1);
        const uint32_t T1 = m1 | e1;
        const uint32_t ca = lop3<kLutAndNot>(a0, T0, 0u), cb = lop3<kLutAndNot>(b0, T0, 0u);  // borrows
        if constexpr (RAMP) {
            const uint32_t mk = (2u << u) - 1u;
            V0 = lop3<kLutXorAnd>(T0, a0, mk);
            V1 = lop3<kLutXor3>(T1, a1, ca) & mk;
        } else {
            V0 = T0 ^ a0;
            V1 = lop3<kLutXor3>(T1, a1, ca);
        }
        H0 = T0 ^ b0;
        H1 = lop3<kLutXor3>(T1, b1, cb);
    }
    Q0 = __funnelshift_l(H0, Q0, 1);
    Q1 = __funnelshift_l(H1, Q1, 1);
}

template <bool GEN, bool RAMP, bool FIRST>
__device__ __forceinline__ void bits_chunk(uint32_t &H0, uint32_t &H1, uint32_t &V0, uint32_t &V1, uint32_t &Q0,
                                           uint32_t &Q1, uint32_t A0, uint32_t A1, uint32_t Rc0, uint32_t Rc1,
                                           uint32_t Rn0, uint32_t Rn1, uint32_t rmask, const BitsScoring &g,
                                           uint32_t X1r, uint32_t X0r) {
#pragma unroll
    for (int u = 0; u < 32; ++u)
        bits_step<GEN, RAMP, FIRST>(u, H0, H1, V0, V1, Q0, Q1, A0, A1, __funnelshift_l(Rn0, Rc0, u),
                                    __funnelshift_l(Rn1, Rc1, u), rmask, g, X1r, X0r);
}

// One stripe of a job, lane by lane: its chunks in order, the words of the
// row above in and of its bottom row out through `rows`.  The B window that
// follows a chunk and the row's words are loaded one chunk ahead.
// FIRST: stripe 0 (nothing comes in; padding rows).
template <bool GEN, bool FIRST>
__device__ __forceinline__ void bits_stripe(const BitsArgs &p, uint32_t C, uint32_t n, int64_t Bg, uint32_t A0,
                                            uint32_t A1, uint32_t rmask, bool last, uint2 *rows, int32_t &W) {
    const uint32_t X1r = p.g.X1 & rmask, X0r = p.g.X0 & rmask;
    uint32_t H0 = 0, H1 = 0, V0 = 0, V1 = 0;
    uint32_t Rc0 = __brev(plane_window(p.pl0, Bg - 31)), Rc1 = __brev(plane_window(p.pl1, Bg - 31));
    uint32_t Fn0 = plane_window(p.pl0, Bg + 1), Fn1 = plane_window(p.pl1, Bg + 1);
    uint2 prev = make_uint2(0u, 0u), nx = make_uint2(0u, 0u);
    if constexpr (!FIRST) {
        prev = __ldcg(rows);
        if (C > 1) nx = __ldcg(rows + 32u);
    }
    for (uint32_t c = 0; c < C; ++c) {
        const uint32_t Rn0 = __brev(Fn0), Rn1 = __brev(Fn1);
        const int64_t gb = Bg + 32 * (int64_t)min(c + 1, C - 1) + 1;
        Fn0 = plane_window(p.pl0, gb);
        Fn1 = plane_window(p.pl1, gb);
        uint32_t Q0 = 0, Q1 = 0;
        if constexpr (!FIRST) {
            // input bits: the previous stripe's bottom row, columns 32c+1 .. 32c+32,
            // column 32c+1 at bit 31
            Q0 = __funnelshift_r(nx.x, prev.x, 1);
            Q1 = __funnelshift_r(nx.y, prev.y, 1);
            prev = nx;
            nx = c + 2 < C ? __ldcg(rows + (size_t)(c + 2) * 32u) : make_uint2(0u, 0u);
        }
        if (c == 0) bits_chunk<GEN, true, FIRST>(H0, H1, V0, V1, Q0, Q1, A0, A1, Rc0, Rc1, Rn0, Rn1, rmask, p.g, X1r, X0r);
        else bits_chunk<GEN, false, FIRST>(H0, H1, V0, V1, Q0, Q1, A0, A1, Rc0, Rc1, Rn0, Rn1, rmask, p.g, X1r, X0r);
        // outgoing bits: bit b is column 32c+1-b of the stripe's bottom row
        if (!last) {
            __stcg(rows + (size_t)c * 32u, make_uint2(Q0, Q1));
        } else {
            const int32_t lo = max(32 * (int32_t)c + 1 - (int32_t)n, 0), hi = min(31, 32 * (int32_t)c);
            if (lo <= hi) {
                const uint32_t mk = (hi == 31 ? ~0u : ((2u << hi) - 1u)) & (~0u << lo);
                W += __popc(Q0 & mk) + 2 * __popc(Q1 & mk);
            }
        }
        Rc0 = Rn0;
        Rc1 = Rn1;
    }
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

template <bool GEN>
__global__ void __launch_bounds__(kBitsWarps * 32) k_bits_score(BitsArgs p) {
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
        const uint32_t S = job.S, C = job.C;
        int32_t W = 0;
        const int64_t Ag = (int64_t)aw * 32 - kPlanePad, Bg = (int64_t)bw * 32 - kPlanePad;  // planar slots
        const int32_t top0 = (int32_t)m - 32 * (int32_t)S;             // row above bit 0 of stripe 0
        for (uint32_t s = 0; s < S; ++s) {
            const int64_t abase = max(Ag + top0 + 32 * (int64_t)s, Ag - 32);
            const uint32_t A0 = plane_window(p.pl0, abase), A1 = plane_window(p.pl1, abase);
            if (s == 0) bits_stripe<GEN, true>(p, C, n, Bg, A0, A1, ~0u << min(max(-top0, 0), 31), S == 1, rows, W);
            else bits_stripe<GEN, false>(p, C, n, Bg, A0, A1, ~0u, s + 1 == S, rows, W);
        }
        if (active) {
            const int32_t sc = W * p.unit + p.gap * (int32_t)(m + n);
            if (in_range(out0, p.score_cap, p.err, kSiteBatchScore)) p.scores[out0] = sc;
            if (out1 != ~0u && in_range(out1, p.score_cap, p.err, kSiteBatchScore)) p.scores[out1] = sc;
        }
    }
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

// Stripes and chunks per stripe of an m x n pair.
static uint32_t stripes_of(uint32_t m) { return (m + 31) / 32; }
static uint32_t chunks_of(uint32_t n) { return (n + 62) / 32; }

// The launch's tables in one upload, its constants, grid and row buffers.
// `head`: the task table, or the sequence and class tables (16-byte padded).
static int bits_finish_plan(nw_ctx *ctx, const uint8_t *pool, std::vector<uint8_t> &head, std::vector<BitsJob> &jobs,
                            uint32_t maxC, const nw_scoring &sc, int32_t *scores, uint32_t score_cap,
                            const std::string &prefix, BitsPlan *plan, void **dhead) {
    int rc;
    // longest jobs first, ties in job order
    std::vector<uint64_t> keys(jobs.size());
    for (size_t q = 0; q < jobs.size(); ++q) keys[q] = (uint64_t)jobs[q].S * jobs[q].C;
    const std::vector<uint32_t> jo = radix_order_desc(std::move(keys));
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
    // their scheduler with the rest and finish the launch alone.  Measured on
    // GB300 (all-vs-all of 512 sequences, CTAs per SM 8 / 3 / 2 / 1): 17.6k /
    // 17.7k / 22.4k / 23.7k GCUPS.  NW_BITS_OCC overrides (sweeps).
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

int bits_prepare(nw_ctx *ctx, const uint8_t *pool, const std::vector<BatchTask> &tasks, const nw_scoring &sc,
                 int32_t *scores, uint32_t score_cap, const std::string &prefix, BitsPlan *plan) {
    *plan = BitsPlan{};
    if (tasks.empty()) return NW_OK;
    HostTimer ht(ctx, "bits_plan");
    // rows: the orientation with fewer stripe-chunks (the score is symmetric);
    // order: equal stripe counts, widest first
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
        turned[k] = (uint64_t)stripes_of(t.n) * chunks_of(t.m) < (uint64_t)stripes_of(t.m) * chunks_of(t.n);
        const uint32_t rows = turned[k] ? t.n : t.m, cols = turned[k] ? t.m : t.n;
        keys[k] = (uint64_t)stripes_of(rows) << 32 | cols;
        bytes += (t.m + 3) / 4 + (t.n + 3) / 4;
        extent = std::max(extent, std::max(t.a_off + (t.m + 3) / 4, t.b_off + (t.n + 3) / 4));
    }
    const std::vector<uint32_t> order = radix_order_desc(std::move(keys));
    // Planar copies: a slot for each of a task's sequences, unless the tasks
    // read their sequences several times over (then the distinct sequences,
    // found by hashing, which costs the host more than the device saves
    // otherwise: 20,000 pairs of distinct reads, 1 ms).
    const bool own = bytes <= 2 * extent;
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
        const uint32_t S = (b.m && b.n) ? stripes_of(b.m) : 0u;
        if (S && own) {
            b.aw = (uint32_t)words;
            b.bw = b.aw + (b.m + 31) / 32 + 2;
            words = (uint64_t)b.bw + (b.n + 31) / 32 + 2;
            if (words >= (1ull << 32)) return fail(ctx, NW_ERR_ARG, "planar copy of more than 2^37 bases");
        } else if (S) {
            b.aw = PlaneSet::word_of(plan->planes.add(b.a_off, b.m));
            b.bw = PlaneSet::word_of(plan->planes.add(b.b_off, b.n));
        }
        ht_[q] = b;
        if (jobs.empty() || jobs.back().S != S || jobs.back().cnt == 32)
            jobs.push_back(BitsJob{(uint32_t)q, 0, S, S ? chunks_of(b.n) : 0, 0});
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
    std::vector<BitsClass> classes;
    std::vector<BitsJob> jobs;
    uint32_t maxC = 1;
    for (uint32_t r0 = 0; r0 < nseq;) {
        const uint32_t S = stripes_of(seqs[r0].len);
        uint32_t r1 = r0;
        while (r1 < nseq && stripes_of(seqs[r1].len) == S) ++r1;
        const uint32_t rows = r1 - r0, pairs = r0 * rows + rows * (rows - 1) / 2;
        // the pairs run through the columns in order: a job's first column is its widest
        uint32_t c = 0;
        auto end_of = [&](uint32_t col) {  // pairs of the columns up to col
            const uint32_t x = col < r0 ? 0u : col - r0 + 1u;
            return col < r0 ? (col + 1u) * rows : r0 * rows + (uint32_t)((uint64_t)x * (2ull * rows - x - 1u) / 2u);
        };
        for (uint32_t q = 0; q < pairs; q += 32) {
            while (end_of(c) <= q) ++c;
            jobs.push_back(BitsJob{q, std::min(32u, pairs - q), S, S ? chunks_of(seqs[c].len) : 0,
                                   (uint32_t)classes.size()});
            maxC = std::max(maxC, jobs.back().C);
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
    cudaMemsetAsync(plan.ba.counter, 0, 4, ctx->stream);
    if (plan.ntasks) {
        LaunchTimer t(ctx, "planes");
        const uint32_t blocks = std::min<uint32_t>((plan.ntasks + 3) / 4, 4096);
        k_planes_tasks<<<blocks, 256, 0, ctx->stream>>>(plan.pool, plan.ba.tasks, plan.ntasks, plan.planes.planes(),
                                                        plan.planes.planes() + plan.planes.plane_words());
    } else if (int rc = plan.planes.enqueue(ctx, plan.pool)) {
        return rc;
    }
    {
        LaunchTimer t(ctx, "bits_score");
        if (plan.gen) k_bits_score<true><<<plan.blocks, kBitsWarps * 32, 0, ctx->stream>>>(plan.ba);
        else k_bits_score<false><<<plan.blocks, kBitsWarps * 32, 0, ctx->stream>>>(plan.ba);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "bit-sliced launch");
}

}  // namespace nw
