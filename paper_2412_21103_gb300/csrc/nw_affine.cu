// Affine gaps (Gotoh; not in the paper, whose gap penalty is linear -- the
// center-star method it cites uses affine gaps): a run of k gap moves of one
// kind scores go + k*ge.  Three grids: E (ends in a horizontal move), F
// (ends in a vertical move), H (best):
//     E(i,j) = max(E(i,j-1) + ge, H(i,j-1) + go + ge)
//     F(i,j) = max(F(i-1,j) + ge, H(i-1,j) + go + ge)
//     H(i,j) = max(H(i-1,j-1) + s(A_i,B_j), E(i,j), F(i,j))
// from H(0,0) = 0, H(0,j) = E(0,j) = go + j*ge, H(i,0) = F(i,0) = go + i*ge.
//
// Shifted domain: W = H - ge*(i+j), E' = E - ge*(i+j), F' = F - ge*(i+j).
// Every move adds one to i+j, so the extension cost drops out:
//     E'(i,j) = max(E'(i,j-1), W(i,j-1) + go)
//     F'(i,j) = max(F'(i-1,j), W(i-1,j) + go)
//     W(i,j)  = max(W(i-1,j-1) + s - 2*ge, E'(i,j), F'(i,j))
// with W(0,0) = 0, W(0,j) = W(i,0) = go, F'(0,j) = E'(i,0) = -inf and
// H(m,n) = W(m,n) + ge*(m+n).  A cell is a score (s - 2ge: from shared
// memory, or a byte permute), two DPX add-max (E', F'), an add and a three-input
// max (W).
//
// Alignments.  The fill writes no pointers: it keeps every stripe's bottom
// row (which the next stripe reads anyway) and, every kTileSteps steps, the
// state of a stripe's 32 lanes.  The trace then walks back from (m, n) tile by
// tile -- a tile is one stripe and the steps between two kept states --
// recomputing only the tiles the path crosses, up to the path's own step,
// with four bits per cell in shared memory: L (the diagonal candidate is below
// max(E', F')), H (E' above F'), and the extension bits of the cell's gap
// states, F: F'(i-1,j) > W(i-1,j) + go, E: E'(i,j-1) > W(i,j-1) + go (a tie
// closes the gap).  Writing the four bits of every cell cost the fill eight
// more operations per cell (13 against 5) and 0.5 bytes.
//
// Batched by stripe jobs: every 32R-row stripe of every pair is one job,
// jobs queued pair by pair (longest pairs first) and stripes in order, so a
// long pair's stripes run on many warps at once as a wavefront instead of
// one after another on one warp (which left a batch waiting on its longest
// pair).  A warp takes the next job from an atomic counter; lane k owns R
// rows of the stripe and a step hands the lane below two values (W with the
// base code, and F').  Every 32 steps the warp writes what lane 31 produced of
// the stripe's bottom row (W and F', through shared memory) to the job's row
// buffer and publishes it with a release store to the job's progress word; the
// warp of the next stripe waits (a bounded spin) on that word before it reads
// a chunk of 32 columns that it has not seen published yet.
// The job it waits on was taken earlier by a warp of the same persistent,
// fully resident grid, so every wait ends.
#include <algorithm>
#include <vector>

#include "nw_internal.cuh"

namespace nw {
namespace {

constexpr int kAffWarps = 8;
constexpr int32_t kAffNeg = -(1 << 27);   // -inf: far below any W, no add wraps
constexpr uint32_t kTileSteps = 128;      // steps between a stripe's kept states
constexpr int kTraceWarps = 3;            // tiles the trace replays at once

struct AffTask {
    uint64_t a_off, b_off;
    uint32_t m, n;
    uint32_t out;
    uint32_t nr;         // words per row half (n rounded up to 32)
    uint64_t row_off;    // word offset of the pair's stripe rows: stripe s (< S-1) at row_off + 2*s*nr
    uint64_t keep_off;   // 16-byte units: the pair's kept states, [stripe][state 1..][part][lane]
    uint32_t keep_n;     // kept states per stripe
    uint32_t pad;
};

struct AffJob {
    uint32_t task;       // index into the launch's tasks
    uint32_t stripe;
};

struct AffArgs {
    const uint8_t *pool;
    const AffTask *tasks;
    const AffJob *jobs;
    uint32_t njobs;
    uint32_t *counter;
    uint32_t prof[4];    // byte d of prof[c] = s(c, d) - 2*ge as int8
    int32_t go, ge;
    uint32_t *rows;      // stripe rows of every pair (W words, then F' words)
    uint64_t rows_cap;
    uint32_t *progress;  // per job: columns of its bottom row published
    int32_t *scores;
    uint4 *keep;         // kept states
    uint64_t keep_cap;
    uint32_t *err;
    uint32_t out_cap;    // pairs at scores (checked build)
};

template <int R>
__device__ __forceinline__ uint32_t aff_rows(const uint8_t *s, uint32_t i0, uint32_t m) {
    uint32_t w = 0;
    if (i0 < m) {
        const uint32_t nbytes = (m + 3) / 4;
#pragma unroll
        for (int q = 0; q < R / 4; ++q) {
            const uint32_t byte = i0 / 4 + q;
            if (byte < nbytes) w |= (uint32_t)__ldg(s + byte) << (8 * q);
        }
    }
    return w;
}

// A lane's R rows of a stripe: the systolic state between two steps.
template <int R>
struct AffLane {
    static constexpr uint32_t kParts = (2 * R + 4) / 4;  // 16-byte parts of a kept state
    uint32_t prof[R];
    int32_t Wl[R], El[R];
    int32_t dtop;        // W of the row above the lane's first, one column back
    uint32_t xout;       // the last row's W (<< 2) and the column's base code, for the lane below
    int32_t fout;        // its F'
    uint32_t accL, accH, accF, accE;

    __device__ __forceinline__ void rows(const AffArgs &p, const uint8_t *A, uint32_t i0, uint32_t m) {
        const uint32_t codes = aff_rows<R>(A, i0, m);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t c = (codes >> (2 * r)) & 3u;
            prof[r] = c == 0 ? p.prof[0] : c == 1 ? p.prof[1] : c == 2 ? p.prof[2] : p.prof[3];
        }
    }
    // column 0: W(i, 0) = go, E'(i, 0) = -inf
    __device__ __forceinline__ void start(int32_t go, uint32_t i0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            Wl[r] = go;
            El[r] = kAffNeg;
        }
        dtop = i0 == 0 ? 0 : go;  // W(i0, 0)
        xout = 0;
        fout = kAffNeg;
    }
    __device__ __forceinline__ void save(uint4 *k, uint64_t cap_left, uint32_t *err) const {
        uint32_t v[4 * kParts];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r] = (uint32_t)Wl[r];
            v[R + r] = (uint32_t)El[r];
        }
        v[2 * R] = (uint32_t)dtop;
        v[2 * R + 1] = xout;
        v[2 * R + 2] = (uint32_t)fout;
        v[2 * R + 3] = 0u;
#pragma unroll
        for (uint32_t q = 0; q < kParts; ++q)
            if (in_range(q * 32u, cap_left, err, kSiteAffPtr))
                __stcg(k + q * 32u, make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
    }
    __device__ __forceinline__ void load(const uint4 *k) {
        uint32_t v[4 * kParts];
#pragma unroll
        for (uint32_t q = 0; q < kParts; ++q) {
            const uint4 x = __ldcg(k + q * 32u);
            v[4 * q] = x.x;
            v[4 * q + 1] = x.y;
            v[4 * q + 2] = x.z;
            v[4 * q + 3] = x.w;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            Wl[r] = (int32_t)v[r];
            El[r] = (int32_t)v[R + r];
        }
        dtop = (int32_t)v[2 * R];
        xout = v[2 * R + 1];
        fout = (int32_t)v[2 * R + 2];
    }
    // The R cells of one column from the row above's word x (W << 2 | code)
    // and F' fx; PTR appends the four bits of each cell to the accumulators
    // (the last R bits of each are this column's, row 0 highest).
    // TAB: the scores of the lane's last kTabRows rows come from shared memory by
    // the column's base, four to a load, not by a byte permute each.
    static constexpr int kTabRows = R >= 8 ? 8 : 0;
    // the lane's table: kTabRows scores for each base of B
    __device__ __forceinline__ void table(int4 *tab) const {
#pragma unroll
        for (uint32_t b = 0; b < 4; ++b)
#pragma unroll
            for (int q = 0; q < kTabRows / 4; ++q) {
                const uint32_t *pr = prof + (R - kTabRows) + 4 * q, sel = sext_selector(b);
                tab[(b * (kTabRows / 4) + q) * 32] = make_int4((int32_t)prmt(pr[0], 0u, sel), (int32_t)prmt(pr[1], 0u, sel),
                                                               (int32_t)prmt(pr[2], 0u, sel), (int32_t)prmt(pr[3], 0u, sel));
            }
    }
    template <bool PTR, bool TAB>
    __device__ __forceinline__ void column(int32_t go, uint32_t x, int32_t fx, const int4 *tab) {
        const uint32_t sel = sext_selector(x & 3u);
        int32_t tv[kTabRows ? kTabRows : 1];
        if constexpr (TAB) {
#pragma unroll
            for (int q = 0; q < kTabRows / 4; ++q) {
                const int4 v = tab[((x & 3u) * (kTabRows / 4) + q) * 32];
                tv[4 * q] = v.x;
                tv[4 * q + 1] = v.y;
                tv[4 * q + 2] = v.z;
                tv[4 * q + 3] = v.w;
            }
        }
        int32_t u = (int32_t)x >> 2, d = dtop, fu = fx;
        dtop = u;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r - (R - kTabRows);
            const int32_t sv = TAB && k >= 0 ? tv[k >= 0 ? k : 0] : (int32_t)prmt(prof[r], 0u, sel);
            const int32_t e = __viaddmax_s32(Wl[r], go, El[r]);
            const int32_t f = __viaddmax_s32(u, go, fu);
            const int32_t w = __vimax3_s32(d + sv, e, f);
            if constexpr (PTR) {
                accL = ptr_append(accL, d + sv - w);
                accH = ptr_append(accH, f - e);
                accF = ptr_append(accF, u + go - fu);
                accE = ptr_append(accE, Wl[r] + go - El[r]);
            }
            d = Wl[r];
            Wl[r] = w;
            El[r] = e;
            u = w;
            fu = f;
        }
        xout = ((uint32_t)u << 2) | (x & 3u);
        fout = fu;
    }
};

// Lane 0's inputs for the columns of a stripe: row 0 (W = go, F' = -inf) for
// stripe 0, else the bottom row of the stripe above.
struct AffAbove {
    const uint8_t *B;
    const uint32_t *inW, *inF;  // null for stripe 0
    uint32_t n;
    int32_t go;
    __device__ __forceinline__ uint32_t w(uint32_t col) const {
        if (col >= n) return 0u;
        if (!inW) return ((uint32_t)go << 2) | base_at(B, col);
        return __ldcg(inW + col);
    }
    __device__ __forceinline__ int32_t f(uint32_t col) const {
        if (!inW || col >= n) return kAffNeg;
        return (int32_t)__ldcg(inF + col);
    }
};

// The fill; KEEP: also the stripes' states every kTileSteps steps (for the
// trace).  What bounds it: the logic pipe, 3 operations per cell (two add-max,
// max3; the add runs on either pipe) and about 12 per column of R cells.
// 2,000 pairs of 1 to 5 kb: 5.2 ms; with a prmt for every row 5.9, for half of
// them 5.55.
template <int R, bool KEEP>
__global__ void __launch_bounds__(kAffWarps * 32) k_affine(AffArgs p) {
    constexpr uint32_t SH = 32u * R;
    const int lane = threadIdx.x & 31;
    const int32_t go = p.go;
    // a chunk's inputs of lane 0 and outputs of lane 31, per warp
    __shared__ uint2 ins_[kAffWarps][32], outs_[kAffWarps][32];
    uint2 *ins = ins_[threadIdx.x >> 5], *outs = outs_[threadIdx.x >> 5];
    constexpr int kTab = 4 * AffLane<R>::kTabRows / 4 * 32;  // a warp's scores, [base][four rows][lane]
    __shared__ int4 tabs_[kTab ? kAffWarps * kTab : 1];
    int4 *tab = tabs_ + (kTab ? (threadIdx.x >> 5) * kTab + lane : 0);

    for (;;) {
        uint32_t jidx = 0;
        if (lane == 0) jidx = atomicAdd(p.counter, 1u);
        jidx = __shfl_sync(kFull, jidx, 0);
        if (jidx >= p.njobs) break;
        const AffJob jb = p.jobs[jidx];
        const AffTask tk = p.tasks[jb.task];
        const uint32_t s = jb.stripe;
        const uint32_t m = tk.m, n = tk.n;
        if (m == 0 || n == 0) {   // a single job
            if (lane == 0 && in_range(tk.out, p.out_cap, p.err, kSiteAffScore))
                p.scores[tk.out] = m + n ? go + p.ge * (int32_t)(m + n) : 0;
            continue;
        }
        const uint32_t S = (m + SH - 1) / SH;
        const uint32_t T = n + 31;
        const uint32_t lM = ((m - 1) % SH) / R, rM = (m - 1) % R;
        // the previous stripe's row (s > 0) and this stripe's (s < S - 1)
        const uint32_t *inW = s ? p.rows + tk.row_off + (size_t)(s - 1) * 2 * tk.nr : nullptr;
        uint32_t *outW = s + 1 < S ? p.rows + tk.row_off + (size_t)s * 2 * tk.nr : nullptr;
        uint32_t *outF = s + 1 < S ? outW + tk.nr : nullptr;
        const uint32_t *prev = s ? p.progress + (jidx - 1) : nullptr;   // stripe s-1 is the job before
        uint32_t *mine = p.progress + jidx;
        const AffAbove above{p.pool + tk.b_off, inW, s ? inW + tk.nr : nullptr, n, go};
        AffLane<R> ln;
        const uint32_t i0 = s * SH + (uint32_t)lane * R;   // rows i0+1 .. i0+R (1-based)
        ln.rows(p, p.pool + tk.a_off, i0, m);
        ln.table(tab);
        ln.start(go, i0);
        uint4 *keep = KEEP ? p.keep + tk.keep_off + (uint64_t)s * tk.keep_n * AffLane<R>::kParts * 32u + lane : nullptr;
        int32_t c = -lane;
        uint32_t seen = 0;
        bool alive = !s || warp_wait_geq(prev, min(32u, n), seen, p.err, jidx);
        uint32_t w_next = alive ? above.w((uint32_t)lane) : 0u;
        int32_t f_next = alive ? above.f((uint32_t)lane) : kAffNeg;
        // the last chunk's bottom row (columns t - 63 .. t - 32 of lane 31) out, and published
        auto row_out = [&](uint32_t t) {
            if (!outW) return;
            __syncwarp();
            const int32_t col = (int32_t)t - 63 + lane;
            if (col >= 0 && col < (int32_t)n &&
                in_range((size_t)(outW - p.rows) + tk.nr + (uint32_t)col, p.rows_cap, p.err, kSiteAffRing)) {
                const uint2 v = outs[lane];
                __stcg(outW + col, v.x);
                __stcg(outF + col, v.y);
            }
            __syncwarp();
            if (lane == 0) st_release(mine, min(t - 31u, n));
        };

        for (uint32_t t = 0; t < T && alive; t += 32) {
            if (KEEP && t && t % kTileSteps == 0) {
                ln.save(keep, p.keep_cap - (uint64_t)(keep - p.keep), p.err);
                keep += AffLane<R>::kParts * 32u;
            }
            __syncwarp();
            ins[lane] = make_uint2(w_next, (uint32_t)f_next);
            __syncwarp();
            if (s && t + 32 < n && !(alive = warp_wait_geq(prev, min(t + 64u, n), seen, p.err, jidx))) break;
            w_next = above.w(t + 32u + (uint32_t)lane);
            f_next = above.f(t + 32u + (uint32_t)lane);
            if (__all_sync(kFull, c >= 0 && c + 32 <= (int32_t)n - 1)) {
#pragma unroll 4
                for (uint32_t uu = 0; uu < 32u; ++uu) {
                    uint32_t x = __shfl_up_sync(kFull, ln.xout, 1);
                    int32_t fx = __shfl_up_sync(kFull, ln.fout, 1);
                    const uint2 in = ins[uu];
                    if (lane == 0) {
                        x = in.x;
                        fx = (int32_t)in.y;
                    }
                    ln.template column<false, true>(go, x, fx, tab);
                    if (lane == 31) outs[uu] = make_uint2(ln.xout, (uint32_t)ln.fout);
                }
                c += 32;
            } else {
                for (uint32_t uu = 0; uu < 32u && t + uu < T; ++uu) {
                    uint32_t x = __shfl_up_sync(kFull, ln.xout, 1);
                    int32_t fx = __shfl_up_sync(kFull, ln.fout, 1);
                    const uint2 in = ins[uu];
                    if (lane == 0) {
                        x = in.x;
                        fx = (int32_t)in.y;
                    }
                    if (c >= 0 && c < (int32_t)n) {
                        ln.template column<false, true>(go, x, fx, tab);
                        if (lane == 31) outs[uu] = make_uint2(ln.xout, (uint32_t)ln.fout);
                        if (s + 1 == S && (uint32_t)lane == lM && c == (int32_t)n - 1) {
                            int32_t wmn = 0;
#pragma unroll
                            for (int r = 0; r < R; ++r)
                                if ((uint32_t)r == rM) wmn = ln.Wl[r];
                            if (in_range(tk.out, p.out_cap, p.err, kSiteAffScore))
                                p.scores[tk.out] = wmn + p.ge * (int32_t)(m + n);
                        }
                    }
                    ++c;
                }
            }
            row_out(t + 32u);
        }
        __syncwarp();
        if (!alive) return;   // a wait gave up (NW_ERR_TIMEOUT is raised): leave
    }
}

// The four bits of a column's R cells as one word: fields L, H, F, E of 8
// bits (R <= 8) or 16 (R = 16), row r at bit R - 1 - r of each field.
template <int R>
struct AffBits {
    using Word = uint32_t;
    __device__ static __forceinline__ Word pack(uint32_t L, uint32_t H, uint32_t F, uint32_t E) {
        return __byte_perm(__byte_perm(L, H, 0x0040), __byte_perm(F, E, 0x0040), 0x5410);
    }
    __device__ static __forceinline__ uint32_t bit(Word w, uint32_t field, uint32_t r) {
        return (w >> (8u * field + (uint32_t)R - 1u - r)) & 1u;
    }
};
template <>
struct AffBits<16> {
    using Word = uint2;
    __device__ static __forceinline__ Word pack(uint32_t L, uint32_t H, uint32_t F, uint32_t E) {
        return make_uint2(__byte_perm(L, H, 0x5410), __byte_perm(F, E, 0x5410));
    }
    __device__ static __forceinline__ uint32_t bit(Word w, uint32_t field, uint32_t r) {
        return ((field < 2 ? w.x : w.y) >> (16u * (field & 1u) + 15u - r)) & 1u;
    }
};

// The walk from (m, n), one CTA per pair, longest pairs first.  The state
// machine: in state H the diagonal when L is clear, else the vertical gap (F)
// when H is clear, else the horizontal one (E); in a gap state the move is
// emitted and the walk stays in the gap while the cell's extension bit is
// set.  Row 0 / column 0: only horizontal / vertical moves remain.  Moves in
// reverse order (0 diagonal, 1 vertical, 2 horizontal).  In state H the warp
// takes a run of diagonal moves at a time: lane q reads the cell q diagonal
// moves on, a ballot of the L bits gives the run; gaps are taken the same way
// (20,000 pairs of 150 and 1,000 bases, mostly one long gap: 4.5 ms, gap moves
// one by one 6.7).
//
// A cell of lane l and column c belongs to step c + l of its stripe; a tile
// holds kTileSteps steps, from a kept state on, and the path's steps only
// fall, so each tile is recomputed once, up to the step of the path's entry.
// The CTA's warps replay kTraceWarps tiles of the path's stripe at once, the one
// of its cell and the ones before it (a path crosses about 2.3 tiles of a
// stripe), then the first warp walks: one warp doing both was bound by its
// longest pair's chain of steps (700 pairs of 1-5 kb 1.7 ms; 2,000 are bound by the
// replayed steps themselves, 2.1 ms either way).
template <int R>
__global__ void __launch_bounds__(32 * kTraceWarps) k_affine_trace(AffArgs p, uint32_t ntasks, uint8_t *moves,
                                                                   const uint64_t *move_off, uint64_t *nmoves) {
    using Bits = AffBits<R>;
    constexpr uint32_t SH = 32u * R;
    extern __shared__ uint4 tiles_[];  // [tile][step][lane]
    __shared__ uint32_t at[3];         // i, j, state between the warps
    typename Bits::Word *tiles = reinterpret_cast<typename Bits::Word *>(tiles_);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const int32_t go = p.go;
    for (uint32_t q = blockIdx.x; q < ntasks; q += gridDim.x) {
        const AffTask tk = p.tasks[q];
        const uint32_t m = tk.m, n = tk.n;
        uint8_t *mv = moves + move_off[q];
        uint32_t i = m, j = n, state = 0;   // state: 0 H, 1 F (vertical gap), 2 E (horizontal gap)
        uint64_t k = 0;
        for (;;) {
            if (threadIdx.x == 0) {
                at[0] = i;
                at[1] = j;
                at[2] = state;
            }
            __syncthreads();
            i = at[0];
            j = at[1];
            state = at[2];
            if (i == 0 || j == 0) break;
            // the tile of cell (i, j) and the ones before it in its stripe
            const uint32_t s = (i - 1) / SH, tc = (j - 1) + ((i - 1) % SH) / R, tl = tc / kTileSteps;
            const uint32_t ntile = min(tl + 1u, (uint32_t)kTraceWarps), t0 = (tl + 1u - ntile) * kTileSteps;
            if (warp < ntile) {
                typename Bits::Word *tile = tiles + warp * kTileSteps * 32u;
                const uint32_t tw = t0 + warp * kTileSteps, te = min(tc, tw + kTileSteps - 1u);
                const uint32_t *inW = s ? p.rows + tk.row_off + (size_t)(s - 1) * 2 * tk.nr : nullptr;
                const AffAbove above{p.pool + tk.b_off, inW, s ? inW + tk.nr : nullptr, n, go};
                AffLane<R> ln;
                const uint32_t i0 = s * SH + lane * R;
                uint32_t stage = 0, stage_next = above.w(tw + lane);
                int32_t fstage = kAffNeg, fstage_next = above.f(tw + lane);
                ln.rows(p, p.pool + tk.a_off, i0, m);
                if (tw)
                    ln.load(p.keep + tk.keep_off +
                            ((uint64_t)s * tk.keep_n + (tw / kTileSteps - 1)) * AffLane<R>::kParts * 32u + lane);
                else
                    ln.start(go, i0);
                ln.accL = ln.accH = ln.accF = ln.accE = 0;
                for (uint32_t t = tw; t <= te; ++t) {
                    if ((t & 31u) == 0) {
                        stage = stage_next;
                        fstage = fstage_next;
                        stage_next = above.w(t + 32u + lane);
                        fstage_next = above.f(t + 32u + lane);
                    }
                    uint32_t x = __shfl_up_sync(kFull, ln.xout, 1);
                    int32_t fx = __shfl_up_sync(kFull, ln.fout, 1);
                    const uint32_t x0 = __shfl_sync(kFull, stage, t & 31u);
                    const int32_t f0 = __shfl_sync(kFull, fstage, t & 31u);
                    if (lane == 0) {
                        x = x0;
                        fx = f0;
                    }
                    if (t >= lane && t - lane < n) {
                        ln.template column<true, false>(go, x, fx, nullptr);
                        tile[(t - tw) * 32u + lane] = Bits::pack(ln.accL, ln.accH, ln.accF, ln.accE);
                    }
                }
            }
            __syncthreads();
            // (uniform over the first warp from here: every lane follows the same walk)
            auto step_of = [&](uint32_t i_, uint32_t j_) { return (j_ - 1) + ((i_ - 1) % SH) / R; };
            while (warp == 0) {
                if (i == 0 || j == 0 || (i - 1) / SH != s || step_of(i, j) < t0) break;
                if (state == 0) {
                    uint32_t stop = 1u, h = 0u;
                    if (lane < i && lane < j) {
                        const uint32_t iq = i - lane, jq = j - lane;
                        if ((iq - 1) / SH == s && step_of(iq, jq) >= t0) {
                            const uint32_t l = ((iq - 1) % SH) / R, r = (iq - 1) % R;
                            const typename Bits::Word w = tiles[(jq - 1 + l - t0) * 32u + l];
                            stop = Bits::bit(w, 0, r);
                            h = stop ? 2u + Bits::bit(w, 1, r) : 0u;  // the gap that ends the run, + 1
                        }
                    }
                    const uint32_t b = __ballot_sync(kFull, stop);
                    const uint32_t run = b ? (uint32_t)__ffs(b) - 1u : 32u;
                    if (lane < run) mv[k + lane] = 0;
                    k += run;
                    i -= run;
                    j -= run;
                    h = __shfl_sync(kFull, h, run & 31u);
                    if (run < 32u && h) state = h - 1u;
                } else {
                    // a run of gap moves: lane q reads the cell q moves on, the
                    // first whose gap does not extend ends it (after its move)
                    const bool vert = state == 1;
                    bool in = false, ext = false;
                    if (lane < (vert ? i : j)) {
                        const uint32_t iq = vert ? i - lane : i, jq = vert ? j : j - lane;
                        if ((iq - 1) / SH == s && step_of(iq, jq) >= t0) {
                            const uint32_t l = ((iq - 1) % SH) / R, r = (iq - 1) % R;
                            in = true;
                            ext = Bits::bit(tiles[(jq - 1 + l - t0) * 32u + l], vert ? 2 : 3, r);
                        }
                    }
                    const uint32_t end = __ballot_sync(kFull, !ext);
                    const uint32_t f = end ? (uint32_t)__ffs(end) - 1u : 32u;
                    const uint32_t closes = f < 32u ? __shfl_sync(kFull, (int)in, f & 31u) : 0u;  // (else it leaves the tiles)
                    const uint32_t run = f + closes;
                    if (lane < run && in_range(k + lane, (uint64_t)m + n, p.err, kSiteAffMoves)) mv[k + lane] = (uint8_t)state;
                    k += run;
                    if (vert) i -= run;
                    else j -= run;
                    if (closes) state = 0;
                }
            }
        }
        if (warp == 0) {
            const uint32_t rest = i + j;
            const uint8_t mvr = i ? 1 : 2;
            for (uint32_t x = lane; x < rest; x += 32) mv[k + x] = mvr;
            if (lane == 0) nmoves[q] = k + rest;
        }
        __syncthreads();
    }
}

template <int R, bool KEEP>
int launch_affine_R(nw_ctx *ctx, AffArgs &aa) {
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_affine<R, KEEP>, kAffWarps * 32, 0);
    if (occ < 1) occ = 1;
    // every CTA resident: a job's warp may wait on an earlier job's warp
    uint32_t blocks = (uint32_t)occ * (uint32_t)ctx->sm_count;
    const uint32_t need = (aa.njobs + kAffWarps - 1) / kAffWarps;
    if (blocks > need) blocks = need ? need : 1;
    void *v = nullptr;
    int rc = scratch(ctx, "affine_counter", 16, &v);
    if (rc) return rc;
    aa.counter = (uint32_t *)v;
    cudaMemsetAsync(aa.counter, 0, 4, ctx->stream);
    LaunchTimer t(ctx, KEEP ? "affine_fill_ptr" : "affine_score");
    k_affine<R, KEEP><<<blocks, kAffWarps * 32, 0, ctx->stream>>>(aa);
    return NW_OK;
}

int launch_affine(nw_ctx *ctx, int R, bool keep, AffArgs &aa) {
    if (keep) {
        if (R == 4) return launch_affine_R<4, true>(ctx, aa);
        if (R == 16) return launch_affine_R<16, true>(ctx, aa);
        return launch_affine_R<8, true>(ctx, aa);
    }
    if (R == 4) return launch_affine_R<4, false>(ctx, aa);
    if (R == 16) return launch_affine_R<16, false>(ctx, aa);
    return launch_affine_R<8, false>(ctx, aa);
}

template <int R>
int launch_affine_trace_R(nw_ctx *ctx, const AffArgs &aa, uint32_t ntasks, uint8_t *moves, const uint64_t *move_off,
                          uint64_t *nmoves) {
    constexpr int smem = kTraceWarps * (int)kTileSteps * 32 * (int)sizeof(typename AffBits<R>::Word);
    if (smem + 64 > 48 * 1024) {  // (with the static words)
        // one value for every caller: the attribute belongs to the process
        const cudaError_t e = cudaFuncSetAttribute(k_affine_trace<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "affine trace shared memory");
    }
    k_affine_trace<R><<<std::min<uint32_t>(ntasks, 65535), 32 * kTraceWarps, smem, ctx->stream>>>(aa, ntasks, moves,
                                                                                               move_off, nmoves);
    return NW_OK;
}

int launch_affine_trace(nw_ctx *ctx, int R, const AffArgs &aa, uint32_t ntasks, uint8_t *moves,
                        const uint64_t *move_off, uint64_t *nmoves) {
    if (R == 4) return launch_affine_trace_R<4>(ctx, aa, ntasks, moves, move_off, nmoves);
    if (R == 16) return launch_affine_trace_R<16>(ctx, aa, ntasks, moves, move_off, nmoves);
    return launch_affine_trace_R<8>(ctx, aa, ntasks, moves, move_off, nmoves);
}

template <typename T>
int aff_upload(nw_ctx *ctx, const char *slot, const std::vector<T> &v, T **dev) {
    void *d = nullptr;
    int rc = to_device(ctx, v.data(), v.size() * sizeof(T), slot, &d);
    if (rc) return rc;
    cudaError_t e = cudaStreamSynchronize(ctx->stream);  // the host vector may be freed right after
    if (e != cudaSuccess) return cuda_fail(ctx, e, "task upload sync");
    *dev = (T *)d;
    return NW_OK;
}

// Stripe jobs of a launch's tasks (in order, stripes in order), the tasks'
// row-buffer offsets, and the row buffers and progress words in scratch.
int affine_jobs(nw_ctx *ctx, std::vector<AffTask> &tasks, int R, AffArgs &aa) {
    const uint32_t SH = 32u * R;
    std::vector<AffJob> jobs;
    uint64_t rows = 0;
    for (uint32_t q = 0; q < tasks.size(); ++q) {
        AffTask &t = tasks[q];
        const uint32_t S = (t.m && t.n) ? (t.m + SH - 1) / SH : 1;
        t.nr = (t.n + 31) / 32 * 32;
        t.row_off = rows;
        rows += (uint64_t)(S - 1) * 2 * t.nr;
        for (uint32_t s = 0; s < S; ++s) jobs.push_back(AffJob{q, s});
    }
    int rc;
    void *rv = nullptr, *pv = nullptr;
    if ((rc = scratch(ctx, "affine_rows", rows * 4 + 16, &rv))) return rc;
    if ((rc = scratch(ctx, "affine_progress", jobs.size() * 4 + 16, &pv))) return rc;
    cudaError_t e = cudaMemsetAsync(pv, 0, jobs.size() * 4, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "affine progress reset");
    AffTask *dt = nullptr;
    AffJob *dj = nullptr;
    if ((rc = aff_upload(ctx, "affine_tasks", tasks, &dt))) return rc;
    if ((rc = aff_upload(ctx, "affine_jobs", jobs, &dj))) return rc;
    aa.tasks = dt;
    aa.jobs = dj;
    aa.njobs = (uint32_t)jobs.size();
    aa.rows = (uint32_t *)rv;
    aa.rows_cap = rows;
    aa.progress = (uint32_t *)pv;
    return NW_OK;
}

int affine_device(nw_ctx *ctx, const uint8_t *pool, const uint64_t *a_off, const uint32_t *a_len,
                  const uint64_t *b_off, const uint32_t *b_len, uint32_t npairs, const nw_affine_scoring &sc,
                  uint32_t flags, int32_t *scores, char *cigar_pool, const uint64_t *cigar_off, uint64_t *cigar_len) {
    const bool want = flags & NW_CIGAR;
    int R = 8;
    if (const char *e = getenv("NW_AFFINE_R")) R = atoi(e) == 4 ? 4 : atoi(e) == 16 ? 16 : 8;
    const uint32_t SH = 32u * R;
    AffArgs aa{};
    aa.pool = pool;
    for (int c = 0; c < 4; ++c) {
        uint32_t w = 0;
        for (int d = 0; d < 4; ++d)
            w |= (uint32_t)(uint8_t)(int8_t)((c == d ? sc.match : sc.mismatch) - 2 * sc.gap_extend) << (8 * d);
        aa.prof[c] = w;
    }
    aa.go = sc.gap_open;
    aa.ge = sc.gap_extend;
    aa.scores = scores;
    aa.err = ctx->d_err;
    aa.out_cap = npairs;
    std::vector<AffTask> all(npairs);
    for (uint32_t k = 0; k < npairs; ++k) {
        AffTask &t = all[k];
        t = AffTask{a_off[k], b_off[k], a_len[k], b_len[k], k, 0, 0, 0, 0, 0};
        // states before steps kTileSteps, 2 kTileSteps, .. of a stripe's n + 31
        if (want && t.m && t.n) t.keep_n = (t.n + 30) / kTileSteps;
    }
    // longest pairs first: their stripe jobs start first
    std::stable_sort(all.begin(), all.end(), [](const AffTask &x, const AffTask &y) {
        return (uint64_t)x.m * x.n > (uint64_t)y.m * y.n;
    });
    int rc;
    if (!want) {
        if ((rc = affine_jobs(ctx, all, R, aa))) return rc;
        return launch_affine(ctx, R, false, aa);
    }
    // Waves that fit a third of the free budget with all they take: kept states,
    // stripe rows, and the moves and tables, which are most of it for short
    // pairs.  A third, because the slots keep the largest size of every wave.
    const uint64_t wave_budget = (ctx->budget - std::min(ctx->budget, ctx->used)) / 3;
    const uint32_t state_units = (2u * (uint32_t)R + 4u) / 4u * 32u;  // 16-byte units of a kept state
    size_t k0 = 0;
    while (k0 < all.size()) {
        std::vector<AffTask> wave;
        std::vector<uint64_t> moff;
        uint64_t units = 0, mbytes = 0, bytes = 0;
        size_t k = k0;
        for (; k < all.size(); ++k) {
            AffTask t = all[k];
            const uint64_t S = (t.m + SH - 1) / SH;
            const uint64_t u = S * t.keep_n * state_units;
            const uint64_t rb = S > 1 ? (S - 1) * 8 * (((uint64_t)t.n + 31) / 32 * 32) : 0;
            const uint64_t more = u * 16 + rb + t.m + t.n + 16 + 2 * sizeof(uint64_t) + sizeof(TraceTask) +
                                  sizeof(AffTask) + std::max<uint64_t>(S, 1) * (sizeof(AffJob) + 4);
            if (!wave.empty() && bytes + more > wave_budget) break;
            bytes += more;
            t.keep_off = units;
            units += u;
            moff.push_back(mbytes);
            mbytes += (uint64_t)t.m + t.n + 16;
            wave.push_back(t);
        }
        void *pv = nullptr, *mv = nullptr, *nm = nullptr;
        if ((rc = scratch(ctx, "affine_keep", units * 16 + 16, &pv))) return rc;
        if ((rc = scratch(ctx, "affine_moves", mbytes + 16, &mv))) return rc;
        if ((rc = scratch(ctx, "affine_nmoves", wave.size() * 8 + 16, &nm))) return rc;
        if ((rc = affine_jobs(ctx, wave, R, aa))) return rc;
        uint64_t *dmoff = nullptr;
        if ((rc = aff_upload(ctx, "affine_move_off", moff, &dmoff))) return rc;
        aa.keep = (uint4 *)pv;
        aa.keep_cap = units;
        if ((rc = launch_affine(ctx, R, true, aa))) return rc;
        {
            LaunchTimer t(ctx, "affine_walk");
            if ((rc = launch_affine_trace(ctx, R, aa, (uint32_t)wave.size(), (uint8_t *)mv, dmoff, (uint64_t *)nm)))
                return rc;
        }
        std::vector<TraceTask> tt(wave.size());
        for (size_t q = 0; q < wave.size(); ++q) {
            const AffTask &t = wave[q];
            TraceTask x{};
            x.m = t.m;
            x.n = t.n;
            x.moves = (uint8_t *)mv + moff[q];
            x.nmoves = (uint64_t *)nm + q;
            x.a = pool + t.a_off;
            x.b = pool + t.b_off;
            x.cigar = cigar_pool + cigar_off[t.out];
            x.cigar_len = cigar_len + t.out;
            x.band_lo = kNoBand;
            tt[q] = x;
        }
        TraceTask *dtt = nullptr;
        if ((rc = aff_upload(ctx, "affine_trace_tasks", tt, &dtt))) return rc;
        if ((rc = launch_finish(ctx, tt[0], dtt, (uint32_t)tt.size(), (flags & NW_CIGAR_M) ? 1u : 0u))) return rc;
        k0 = k;
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "affine launch");
}

uint64_t aff_pool_extent(const uint64_t *a_off, const uint32_t *a_len, const uint64_t *b_off, const uint32_t *b_len,
                         uint32_t npairs) {
    uint64_t b = 16;
    for (uint32_t k = 0; k < npairs; ++k) {
        b = std::max<uint64_t>(b, a_off[k] + (a_len[k] + 3) / 4);
        b = std::max<uint64_t>(b, b_off[k] + (b_len[k] + 3) / 4);
    }
    return b;
}

}  // namespace
}  // namespace nw

using namespace nw;

extern "C" int nw_affine_align_batch(nw_ctx *ctx, const uint8_t *pool2b, const uint64_t *a_off,
                                     const uint32_t *a_len, const uint64_t *b_off, const uint32_t *b_len,
                                     uint32_t npairs, nw_affine_scoring sc, uint32_t flags, int32_t *scores,
                                     char *cigar_pool, const uint64_t *cigar_off, uint64_t *cigar_len) {
    if (!ctx) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    auto in = [](int v) { return v >= -40 && v <= 40; };
    if (!in(sc.match) || !in(sc.mismatch) || !in(sc.gap_open) || !in(sc.gap_extend))
        return fail(ctx, NW_ERR_ARG, "scores must lie in [-40, 40]");
    if (sc.gap_open > 0 || sc.gap_extend > 0) return fail(ctx, NW_ERR_ARG, "gap open and extend must be <= 0");
    if (sc.mismatch > sc.match) return fail(ctx, NW_ERR_ARG, "mismatch must be <= match");
    if (npairs == 0) return NW_OK;
    const bool want = flags & NW_CIGAR;
    if (!pool2b || !a_off || !a_len || !b_off || !b_len || !scores) return fail(ctx, NW_ERR_ARG, "null argument");
    if (want && (!cigar_pool || !cigar_off || !cigar_len)) return fail(ctx, NW_ERR_ARG, "CIGAR buffers are null");
    const uint64_t sp = sc.match > 2 * sc.gap_extend ? (uint64_t)(sc.match - 2 * sc.gap_extend) : 0;
    for (uint32_t k = 0; k < npairs; ++k) {
        if (a_len[k] >= (1u << 30) || b_len[k] >= (1u << 30)) return fail(ctx, NW_ERR_ARG, "sequence longer than 2^30");
        if (sp * std::min(a_len[k], b_len[k]) >= (1ull << 29))
            return fail(ctx, NW_ERR_ARG, "(match - 2*gap_extend) * min(m,n) must stay below 2^29");
        if (want && cigar_off[k + 1] - cigar_off[k] < nw_cigar_bound(a_len[k], b_len[k]))
            return fail(ctx, NW_ERR_ARG, "CIGAR capacity of pair %u below nw_cigar_bound", k);
    }
    if (!(flags & NW_HOST_IO))
        return affine_device(ctx, pool2b, a_off, a_len, b_off, b_len, npairs, sc, flags, scores, cigar_pool,
                             cigar_off, cigar_len);
    int rc;
    void *dp = nullptr, *ds = nullptr, *dc = nullptr, *dl = nullptr;
    if ((rc = to_device(ctx, pool2b, aff_pool_extent(a_off, a_len, b_off, b_len, npairs), "hio_pool", &dp))) return rc;
    if ((rc = scratch(ctx, "hio_scores", (size_t)npairs * 4, &ds))) return rc;
    if (want) {
        if ((rc = scratch(ctx, "hio_cigar", cigar_off[npairs] + 16, &dc))) return rc;
        if ((rc = scratch(ctx, "hio_cigar_len", (size_t)npairs * 8, &dl))) return rc;
    }
    if ((rc = affine_device(ctx, (const uint8_t *)dp, a_off, a_len, b_off, b_len, npairs, sc, flags, (int32_t *)ds,
                            (char *)dc, cigar_off, (uint64_t *)dl)))
        return rc;
    cudaError_t e = cudaMemcpyAsync(scores, ds, (size_t)npairs * 4, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && want) e = cudaMemcpyAsync(cigar_len, dl, (size_t)npairs * 8, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && want)
        e = cudaMemcpyAsync(cigar_pool, dc, cigar_off[npairs], cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "affine D2H");
    return nw_ctx_sync(ctx);
}
