// Local alignment (Smith-Waterman; not in the paper): the Sec. 2.3 grid with
// a floor of 0, so an alignment may start and end anywhere:
//     H(i,0) = H(0,j) = 0,
//     H(i,j) = max(0, H(i-1,j-1) + s(A_i,B_j), H(i-1,j) + gap, H(i,j-1) + gap).
// The score is the largest H; the alignment ends at the first cell in
// row-major order holding it and is walked back with the priority diagonal >
// vertical > horizontal until a cell whose H is 0 (its start).
//
// The floor rules out the W domain of the global kernels (it would turn into
// a floor that grows along every anti-diagonal), so the cell works on H itself:
// with G = H + gap kept beside H, one cell is a score (a byte permute, or a word
// from shared memory), two adds (H_diag + s, and G) and one DPX three-input max
// with ReLU, max(H_diag + s, G_up, G_left, 0), and half a three-input max for
// the largest H.
//
// Batched by stripe jobs: every 32R-row stripe of every pair is one job, jobs
// queued pair by pair (longest pairs first) and stripes in order, so a pair's
// stripes run on several warps at once as a wavefront (one warp per pair left
// the launch waiting on its longest pairs).  A warp takes the next job from an
// atomic counter; lane k owns R rows of the stripe.  Every 32 steps the warp
// writes what lane 31 produced of the stripe's bottom row (through shared
// memory) to the pair's row buffer and publishes it with a release store; the
// warp of the next stripe waits (a bounded spin) on that word before it reads a
// chunk of 32 columns that it has not seen published yet.  The job it waits on
// was taken earlier by a warp of the same fully resident grid, so every wait
// ends.
//
// End cells and alignments.  The fill keeps no pointers and no positions: a
// lane notes the first and the last chunk of steps in which its rows reached
// their largest H, and every kTileSteps steps the state of a stripe's lanes is
// kept, with the largest H of the steps since the last one.  The trace finds the
// pair's best lane, recomputes the tiles that reach its largest H for the
// first cell in row-major order, and walks back from it tile by tile -- a tile
// is one stripe and the steps between two kept states -- recomputing only the
// tiles the path crosses (a warp each) with the two pointer bits in shared
// memory (L: the diagonal candidate is below max(up, left) + gap; H: left above
// up), and tracking H along the path to find the start.  Pointers and positions for
// every cell cost the fill 11 operations per cell, against 4.5.
#include <algorithm>
#include <vector>

#include "nw_internal.cuh"
#include "nw_order.h"

namespace nw {
namespace {

constexpr int kLocalWarps = 8;
constexpr uint32_t kLocalMinPeriod = 96;   // columns a stripe counts at least (the limit on a pair's size)
constexpr uint32_t kTileSteps = 128;       // steps between a stripe's kept states
constexpr int kTraceWarps = 3;             // tiles the trace replays at once
// End cells without alignments: pairs of up to this many stripes keep states as
// well.  Replaying a whole stripe on one warp takes about as long as the fill's
// one stripe (1,000 pairs of 200 bases and 200 kb: 33 ms beside a fill of 22, with
// states .25); from a dozen stripes on it is a quarter of the fill, and the
// states would be most of the scratch.
constexpr uint32_t kEndStripes = 4;
constexpr uint32_t kPadProfile = 0x80808080u;  // rows past the end: s = -128, never above a real row

struct LocalTask {
    uint64_t a_off, b_off;
    uint32_t m, n;
    uint32_t out;        // pair index
    uint32_t job0;       // its first stripe job
    uint32_t nr;         // words per stripe row (n rounded up to 32)
    uint32_t keep_n;     // kept states per stripe
    uint64_t row_off;    // word offset of the pair's stripe rows
    uint64_t keep_off;   // 16-byte units: its kept states, [stripe][state 1..][part][lane]
};

struct LocalJob {
    uint32_t task, stripe;
};

// The largest H of a stripe: the first lane that reached it, and the first
// and the last chunk of 32 steps (in a fill that keeps states: tile) in which it did.
struct LocalBest {
    int32_t v;
    uint32_t lane, t0, t1;
};

// What a launch produces: the scores alone, also the stripes' best lanes
// (end cells), or also the kept states and all rows (alignments).
enum LocalMode { kScore = 0, kEnds = 1, kKeep = 2 };

struct LocalArgs {
    const uint8_t *pool;
    const LocalTask *tasks;
    const LocalJob *jobs;
    uint32_t njobs;
    uint32_t *counter;
    uint32_t prof[4];    // byte d of prof[c] = s(c, d) as int8
    int32_t match, mismatch, gap;
    uint32_t *rows;      // stripe rows (H << 2 | base code): all of a pair's, or two in turn (turn)
    uint32_t turn;
    uint64_t rows_cap;
    uint32_t *progress;  // per job: columns of its bottom row published
    LocalBest *best;     // per job
    int32_t *scores;     // [out]
    uint32_t *ends;      // [4*out]: i_start, j_start, i_end, j_end
    uint4 *keep;
    uint64_t keep_cap;
    uint32_t *err;
    uint32_t out_cap;    // pairs at scores / ends (checked build)
};

template <int R>
__device__ __forceinline__ uint32_t rows_codes(const uint8_t *s, uint32_t i0, uint32_t m) {
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
struct LocalLane {
    static constexpr uint32_t kParts = (R + 5) / 4;  // 16-byte parts of a kept state
    static_assert(R % 4 == 0 && R + 2 < 4 * kParts, "the top is the third word of the last part");
    uint32_t prof[R];
    int32_t Hl[R], Gl[R];  // H of the column before, and with the gap's score added (in the fill)
    int32_t dtop;        // H of the row above the lane's first, one column back
    uint32_t xout;       // the last row's H (<< 2) and the column's base code, for the lane below
    uint32_t accL, accH;

    __device__ __forceinline__ void rows(const LocalArgs &p, const uint8_t *A, uint32_t i0, uint32_t m) {
        const uint32_t codes = rows_codes<R>(A, i0, m);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t c = (codes >> (2 * r)) & 3u;
            prof[r] = i0 + r >= m ? kPadProfile
                                  : c == 0 ? p.prof[0] : c == 1 ? p.prof[1] : c == 2 ? p.prof[2] : p.prof[3];
        }
    }
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
    __device__ __forceinline__ void start(int32_t g) {  // column 0
#pragma unroll
        for (int r = 0; r < R; ++r) {
            Hl[r] = 0;
            Gl[r] = g;
        }
        dtop = 0;
        xout = 0;
    }
    // top: the largest H of the lane's rows in the tile that ends here
    __device__ __forceinline__ void save(uint4 *k, int32_t top, uint64_t cap_left, uint32_t *err) const {
        uint32_t v[4 * kParts] = {};
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = (uint32_t)Hl[r];
        v[R] = (uint32_t)dtop;
        v[R + 1] = xout;
        v[R + 2] = (uint32_t)top;
#pragma unroll
        for (uint32_t q = 0; q < kParts; ++q)
            if (in_range(q * 32u, cap_left, err, kSiteLocalPtr))
                __stcg(k + q * 32u, make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
    }
    __device__ __forceinline__ void load(const uint4 *k, int32_t g) {
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
            Hl[r] = (int32_t)v[r];
            Gl[r] = Hl[r] + g;
        }
        dtop = (int32_t)v[R];
        xout = v[R + 1];
    }
    // The R cells of one column from the row above's word x (H << 2 | code);
    // cm takes the largest H.  PTR appends the two bits of each cell to the
    // accumulators (the last R bits of each are this column's, row 0 highest).
    // TAB: the scores of the lane's last kTabRows rows come from shared memory by
    // the column's base, four to a load, not by a byte permute each.
    static constexpr int kTabRows = R >= 8 ? 8 : 0;
    template <bool PTR, bool TAB>
    __device__ __forceinline__ void column(int32_t g, uint32_t x, int32_t &cm, const int4 *tab) {
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
        int32_t u = (int32_t)x >> 2, d = dtop, ug = u + g;
        dtop = u;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r - (R - kTabRows);
            const int32_t sv = TAB && k >= 0 ? tv[k >= 0 ? k : 0] : (int32_t)prmt(prof[r], 0u, sel);
            const int32_t l = Hl[r];
            if constexpr (PTR) {
                const int32_t mg = max(u, l) + g;
                accL = ptr_append(accL, d + sv - mg);
                accH = ptr_append(accH, u - l);
                Hl[r] = __viaddmax_s32_relu(d, sv, mg);
                Gl[r] = Hl[r] + g;
            } else {
                Hl[r] = __vimax3_s32_relu(d + sv, ug, Gl[r]);
                ug = Gl[r] = Hl[r] + g;
                if (r & 1) cm = __vimax3_s32(cm, u, Hl[r]);
            }
            d = l;
            u = Hl[r];
        }
        xout = ((uint32_t)u << 2) | (x & 3u);
    }
};

// Lane 0's inputs for the columns of a stripe: row 0 (H = 0) for stripe 0,
// else the bottom row of the stripe above.
struct LocalAbove {
    const uint8_t *B;
    const uint32_t *in;  // null for stripe 0
    uint32_t n;
    __device__ __forceinline__ uint32_t word(uint32_t col) const {
        if (col >= n) return 0u;
        return in ? __ldcg(in + col) : base_at(B, col);
    }
};

// The fill.  What bounds it: the logic pipe, 1.5 operations per cell (max3,
// half a max3; the adds run on either pipe) and about ten per column of R
// cells, and waits for the stripe above.  4,000 pairs of 2 to 10 kb: 9.8 ms;
// with max, add and add-max per cell (3.5 operations) 12.4, with a prmt for
// every row 10.7, for half of them 10.3.
template <int R, int MODE, bool TAB>
__global__ void __launch_bounds__(kLocalWarps * 32) k_local(LocalArgs p) {
    constexpr uint32_t SH = 32u * R;
    const int lane = threadIdx.x & 31;
    const int32_t g = p.gap;
    // a chunk's inputs of lane 0 and outputs of lane 31, per warp
    __shared__ uint32_t ins_[kLocalWarps][32], outs_[kLocalWarps][32];
    uint32_t *ins = ins_[threadIdx.x >> 5], *outs = outs_[threadIdx.x >> 5];
    constexpr int kTab = TAB ? 4 * LocalLane<R>::kTabRows / 4 * 32 : 0;  // a warp's scores, [base][four rows][lane]
    __shared__ int4 tabs_[kTab ? kLocalWarps * kTab : 1];
    int4 *tab = tabs_ + (kTab ? (threadIdx.x >> 5) * kTab + lane : 0);

    for (;;) {
        uint32_t jidx = 0;
        if (lane == 0) jidx = atomicAdd(p.counter, 1u);
        jidx = __shfl_sync(kFull, jidx, 0);
        if (jidx >= p.njobs) break;
        const LocalJob jb = p.jobs[jidx];
        const LocalTask tk = p.tasks[jb.task];
        const uint32_t s = jb.stripe, m = tk.m, n = tk.n, keep_n = MODE == kKeep ? tk.keep_n : 0u;
        if (m == 0 || n == 0) {  // a single job: the score stays 0
            if (MODE != kScore && lane == 0) p.best[jidx] = LocalBest{0, 0u, 0u, 0u};
            continue;
        }
        const uint32_t S = (m + SH - 1) / SH;
        const uint32_t T = n + 31;
        // rows: all kept, or two in turn (the stripe below has read a column
        // of the row before this one when this stripe's successor overwrites it)
        auto row = [&](uint32_t q) { return p.rows + tk.row_off + (size_t)(p.turn ? q & 1u : q) * tk.nr; };
        const uint32_t *in = s ? row(s - 1) : nullptr;
        uint32_t *out = s + 1 < S ? row(s) : nullptr;
        const uint32_t *prev = s ? p.progress + (jidx - 1) : nullptr;  // stripe s-1 is the job before
        uint32_t *mine = p.progress + jidx;
        const LocalAbove above{p.pool + tk.b_off, in, n};
        LocalLane<R> ln;
        const uint32_t i0 = s * SH + (uint32_t)lane * R;
        ln.rows(p, p.pool + tk.a_off, i0, m);
        if constexpr (TAB) ln.table(tab);
        ln.start(p.gap);
        uint4 *keep = MODE == kKeep ? p.keep + tk.keep_off + (uint64_t)s * tk.keep_n * LocalLane<R>::kParts * 32u + lane
                                    : nullptr;
        int32_t best = 0, cm = 0;    // the lane's largest H before and in this chunk of 32 steps, or tile
        int32_t top = 0;             // ... in the last tile
        uint32_t bt = 0, bl = 0;     // the first and the last chunk or tile that reached it
        int32_t c = -lane;
        uint32_t seen = 0;
        bool alive = !s || warp_wait_geq(prev, min(32u, n), seen, p.err, jidx);
        uint32_t next = alive ? above.word((uint32_t)lane) : 0u;
        // the last chunk's bottom row (columns t - 63 .. t - 32 of lane 31) out, and published
        auto row_out = [&](uint32_t t) {
            if (!out) return;
            __syncwarp();
            const int32_t col = (int32_t)t - 63 + lane;
            if (col >= 0 && col < (int32_t)n &&
                in_range((size_t)(out - p.rows) + (uint32_t)col, p.rows_cap, p.err, kSiteLocalRing))
                __stcg(out + col, outs[lane]);
            __syncwarp();
            if (lane == 0) st_release(mine, min(t - 31u, n));
        };
        for (uint32_t t = 0; t < T && alive; t += 32) {
            if (MODE == kKeep && keep_n && t && t % kTileSteps == 0) {
                ln.save(keep, top, p.keep_cap - (uint64_t)(keep - p.keep), p.err);
                keep += LocalLane<R>::kParts * 32u;
            }
            __syncwarp();
            ins[lane] = next;
            __syncwarp();
            if (s && t + 32 < n && !(alive = warp_wait_geq(prev, min(t + 64u, n), seen, p.err, jidx))) break;
            next = above.word(t + 32u + (uint32_t)lane);
            if (__all_sync(kFull, c >= 0 && c + 32 <= (int32_t)n - 1)) {
#pragma unroll 4
                for (uint32_t uu = 0; uu < 32u; ++uu) {
                    uint32_t x = __shfl_up_sync(kFull, ln.xout, 1);
                    const uint32_t in = ins[uu];
                    if (lane == 0) x = in;
                    ln.template column<false, TAB>(g, x, cm, tab);
                    if (lane == 31) outs[uu] = ln.xout;
                }
                c += 32;
            } else {
                for (uint32_t uu = 0; uu < 32u && t + uu < T; ++uu) {
                    uint32_t x = __shfl_up_sync(kFull, ln.xout, 1);
                    const uint32_t in = ins[uu];
                    if (lane == 0) x = in;
                    if (c >= 0 && c < (int32_t)n) {
                        ln.template column<false, TAB>(g, x, cm, tab);
                        if (lane == 31) outs[uu] = ln.xout;
                    }
                    ++c;
                }
            }
            row_out(t + 32u);
            // (with states a tile at a time: once a chunk took 1% of the fill)
            if (MODE == kEnds || (MODE == kKeep && ((t + 32) % kTileSteps == 0 || t + 32 >= T))) {
                const uint32_t from = MODE == kKeep ? t - t % kTileSteps : t;
                if (cm > best) bt = from;
                if (cm >= best) bl = from;
                best = max(best, cm);
                top = cm;
                cm = 0;
            }
        }
        if (!alive) return;   // a wait gave up (NW_ERR_TIMEOUT is raised): leave
        if (MODE == kScore) best = cm;
        // the stripe's largest H and its first lane
        const int32_t most = __reduce_max_sync(kFull, best);
        if (lane == 0 && most > 0 && in_range(tk.out, p.out_cap, p.err, kSiteLocalOut)) atomicMax(p.scores + tk.out, most);
        if (MODE != kScore) {
            const uint32_t first = (uint32_t)__ffs(__ballot_sync(kFull, best == most)) - 1u;
            if ((uint32_t)lane == first) p.best[jidx] = LocalBest{most, first, bt, bl};
        }
        __syncwarp();
    }
}

// The two bits of a column's R cells: fields L, H of 8 bits (R <= 8) or 16.
template <int R>
struct LocalBits {
    using Word = uint16_t;
    __device__ static __forceinline__ Word pack(uint32_t L, uint32_t H) { return (Word)__byte_perm(L, H, 0x0040); }
    __device__ static __forceinline__ uint32_t bit(Word w, uint32_t field, uint32_t r) {
        return ((uint32_t)w >> (8u * field + (uint32_t)R - 1u - r)) & 1u;
    }
};
template <>
struct LocalBits<16> {
    using Word = uint32_t;
    __device__ static __forceinline__ Word pack(uint32_t L, uint32_t H) { return __byte_perm(L, H, 0x5410); }
    __device__ static __forceinline__ uint32_t bit(Word w, uint32_t field, uint32_t r) {
        return (w >> (16u * field + 15u - r)) & 1u;
    }
};

// A stripe's lanes again, from step t0 (a kept state, or its start) on.
template <int R>
struct LocalReplay {
    LocalLane<R> ln;
    LocalAbove above;
    uint32_t t, stage, stage_next;
    __device__ void begin(const LocalArgs &p, const LocalTask &tk, uint32_t s, uint32_t t0, uint32_t lane) {
        constexpr uint32_t SH = 32u * R;
        const uint32_t in = p.turn ? (s - 1) & 1u : s - 1;
        above = LocalAbove{p.pool + tk.b_off, s ? p.rows + tk.row_off + (size_t)in * tk.nr : nullptr, tk.n};
        t = t0;
        stage = 0;
        stage_next = above.word(t0 + lane);
        ln.rows(p, p.pool + tk.a_off, s * SH + lane * R, tk.m);
        ln.accL = ln.accH = 0;
        if (t0)
            ln.load(p.keep + tk.keep_off +
                    ((uint64_t)s * tk.keep_n + (t0 / kTileSteps - 1)) * LocalLane<R>::kParts * 32u + lane, p.gap);
        else
            ln.start(p.gap);
    }
    // one step; whether the lane had a column
    template <bool PTR>
    __device__ __forceinline__ bool step(int32_t g, uint32_t lane) {
        if ((t & 31u) == 0) {
            stage = stage_next;
            stage_next = above.word(t + 32u + lane);
        }
        uint32_t x = __shfl_up_sync(kFull, ln.xout, 1);
        const uint32_t x0 = __shfl_sync(kFull, stage, t & 31u);
        if (lane == 0) x = x0;
        const bool act = t >= lane && t - lane < above.n;
        int32_t cm = 0;
        if (act) ln.template column<PTR, false>(g, x, cm, nullptr);
        ++t;
        return act;
    }
};

// End cells and, with WALK, the walk back from them: one CTA per pair,
// longest pairs first.  WALK: its warps replay kTraceWarps tiles of the path's
// stripe at once, the one of its cell and the ones before it (a path crosses
// about 2.3 tiles of a stripe), then the first warp follows the path to the first cell whose H is 0;
// moves in reverse order (0 diagonal, 1 vertical, 2 horizontal).  A run of
// diagonal moves is taken at a time: lane q reads the cell q diagonal moves
// on, and H there follows from the matches before it (a ballot).  A pair without
// kept states (of end cells alone, or of few columns) replays its stripe from
// the start.
//
// Where the best lane reaches its largest H again far on -- a read against a long
// reference, one stripe of many tiles -- only the tiles that do are replayed:
// 1,000 pairs of 200 bases and 200 kb .18 ms of trace, with every step from the
// first to the last of them 35.
template <int R, bool WALK>
__global__ void __launch_bounds__(WALK ? 32 * kTraceWarps : 32) k_local_trace(LocalArgs p, uint32_t ntasks,
                                                                              uint8_t *moves, const uint64_t *move_off,
                                                                              uint64_t *nmoves) {
    using Bits = LocalBits<R>;
    constexpr uint32_t SH = 32u * R;
    extern __shared__ uint4 tiles_[];  // [tile][step][lane]
    __shared__ int32_t at[3];          // i, j, h between the warps
    __shared__ uint32_t first_[R];
    typename Bits::Word *tiles = reinterpret_cast<typename Bits::Word *>(tiles_);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    for (uint32_t q = blockIdx.x; q < ntasks; q += gridDim.x) {
        const LocalTask tk = p.tasks[q];
        const uint32_t m = tk.m, n = tk.n, S = (m && n) ? (m + SH - 1) / SH : 1u;
        // the first stripe with the largest H
        int32_t bv = 0;
        uint32_t bs = 0;
        for (uint32_t s0 = 0; s0 < S; s0 += 32) {
            const int32_t v = s0 + lane < S ? p.best[tk.job0 + s0 + lane].v : 0;
            const int32_t top = __reduce_max_sync(kFull, v);
            if (top > bv) {
                bv = top;
                bs = s0 + (uint32_t)__ffs(__ballot_sync(kFull, v == top)) - 1u;
            }
        }
        uint32_t i = 0, j = 0;
        LocalReplay<R> rp;
        if (bv > 0) {
            // the first cell in row-major order among the best lane's rows
            const LocalBest b = p.best[tk.job0 + bs];
            const uint32_t lo = b.t0, hi = min(b.t1 + (p.keep ? kTileSteps : 32u), n + 31u);
            uint32_t first[R];  // by row, the first column found
#pragma unroll
            for (int r = 0; r < R; ++r) first[r] = ~0u;
            const auto look = [&](uint32_t end) {
                while (rp.t < end) {
                    const uint32_t t = rp.t;
                    const bool act = rp.template step<false>(p.gap, lane);
                    if (act && t >= lo && lane == b.lane) {
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            if (rp.ln.Hl[r] == bv && first[r] == ~0u) first[r] = t - lane;
                    }
                }
            };
            if (threadIdx.x < (uint32_t)R) first_[threadIdx.x] = ~0u;
            __syncthreads();
            if (p.keep && tk.keep_n) {
                // the tiles that reach the largest H, dealt out to the warps
                constexpr uint32_t kParts = LocalLane<R>::kParts;
                const uint4 *tops = p.keep + tk.keep_off + ((uint64_t)bs * tk.keep_n * kParts + kParts - 1u) * 32u + b.lane;
                const uint32_t last = b.t1 / kTileSteps;
                uint32_t turn = 0;
                for (uint32_t k0 = lo / kTileSteps; k0 <= last; k0 += 32) {
                    const uint32_t tl = k0 + lane;
                    const bool has = tl == last || (tl < last && (int32_t)__ldcg(tops + (size_t)tl * (kParts * 32u)).z == bv);
                    for (uint32_t todo = __ballot_sync(kFull, has); todo; todo &= todo - 1u)
                        if (turn++ % (blockDim.x >> 5) == warp) {
                            const uint32_t t0 = (k0 + (uint32_t)__ffs(todo) - 1u) * kTileSteps;
                            rp.begin(p, tk, bs, t0, lane);
                            look(min(t0 + kTileSteps, hi));
                        }
                }
            } else {
                // no states: the stripe from its start, and where only two rows
                // are kept (the rows above were overwritten) the stripes above it
                for (uint32_t s = 0; p.turn && s < bs; ++s) {
                    rp.begin(p, tk, s, 0u, lane);
                    uint32_t *out = p.rows + tk.row_off + (size_t)(s & 1u) * tk.nr;
                    while (rp.t < n + 31u) {
                        const uint32_t t = rp.t;
                        if (rp.template step<false>(p.gap, lane) && lane == 31) __stcg(out + (t - 31u), rp.ln.xout);
                    }
                    __threadfence();
                    __syncwarp();
                }
                rp.begin(p, tk, bs, 0u, lane);
                look(hi);
            }
            if (lane == b.lane) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (first[r] != ~0u) atomicMin(&first_[r], first[r]);
            }
            __syncthreads();
#pragma unroll
            for (int r = R - 1; r >= 0; --r)
                if (first_[r] != ~0u) {
                    i = bs * SH + b.lane * R + (uint32_t)r + 1u;
                    j = first_[r] + 1u;
                }
        }
        if (threadIdx.x == 0 && in_range(tk.out, p.out_cap, p.err, kSiteLocalOut)) {
            p.ends[4 * (size_t)tk.out + 2] = i;
            p.ends[4 * (size_t)tk.out + 3] = j;
            if (!WALK) p.ends[4 * (size_t)tk.out + 0] = p.ends[4 * (size_t)tk.out + 1] = ~0u;  // not computed
        }
        if constexpr (WALK) {
            const uint8_t *A = p.pool + tk.a_off, *B = p.pool + tk.b_off;
            uint8_t *mv = moves + move_off[q];
            int32_t h = bv;
            uint64_t k = 0;
            for (;;) {
                if (threadIdx.x == 0) {
                    at[0] = (int32_t)i;
                    at[1] = (int32_t)j;
                    at[2] = h;
                }
                __syncthreads();
                i = (uint32_t)at[0];
                j = (uint32_t)at[1];
                h = at[2];
                if (!(h > 0 && i > 0 && j > 0)) break;
                // the tile of cell (i, j) and the ones before it in its stripe
                const uint32_t s = (i - 1) / SH, tc = (j - 1) + ((i - 1) % SH) / R, tl = tc / kTileSteps;
                const uint32_t ntile = min(tl + 1u, (uint32_t)kTraceWarps), t0 = (tl + 1u - ntile) * kTileSteps;
                if (warp < ntile) {
                    typename Bits::Word *tile = tiles + warp * kTileSteps * 32u;
                    const uint32_t tw = t0 + warp * kTileSteps, te = min(tc, tw + kTileSteps - 1u);
                    rp.begin(p, tk, s, tw, lane);
                    while (rp.t <= te) {
                        const uint32_t t = rp.t;
                        if (rp.template step<true>(p.gap, lane))
                            tile[(t - tw) * 32u + lane] = Bits::pack(rp.ln.accL, rp.ln.accH);
                    }
                }
                __syncthreads();
                // (uniform over the first warp from here: every lane follows the same walk)
                auto step_of = [&](uint32_t i_, uint32_t j_) { return (j_ - 1) + ((i_ - 1) % SH) / R; };
                while (warp == 0 && h > 0 && i > 0 && j > 0 && (i - 1) / SH == s && step_of(i, j) >= t0) {
                    uint32_t stop = 1u, gapm = 0u, same = 0u;
                    if (lane < i && lane < j) {
                        const uint32_t iq = i - lane, jq = j - lane;
                        if ((iq - 1) / SH == s && step_of(iq, jq) >= t0) {
                            const uint32_t l = ((iq - 1) % SH) / R, r = (iq - 1) % R;
                            const typename Bits::Word w = tiles[(jq - 1 + l - t0) * 32u + l];
                            stop = Bits::bit(w, 0, r);
                            gapm = stop ? 1u + Bits::bit(w, 1, r) : 0u;  // the gap move that ends the run
                            same = base_at(A, iq - 1) == base_at(B, jq - 1);
                        }
                    }
                    const uint32_t eq = __ballot_sync(kFull, same), before = (1u << lane) - 1u;
                    const int32_t ne = __popc(eq & before);
                    const int32_t hq = h - p.match * ne - p.mismatch * ((int32_t)lane - ne);  // H of the lane's cell
                    const uint32_t b = __ballot_sync(kFull, stop || hq == 0);
                    const uint32_t run = b ? (uint32_t)__ffs(b) - 1u : 32u;
                    if (lane < run && in_range(k + lane, (uint64_t)m + n, p.err, kSiteLocalMoves)) mv[k + lane] = 0;
                    k += run;
                    i -= run;
                    j -= run;
                    const uint32_t lm = run < 32u ? (1u << run) - 1u : kFull;
                    const int32_t nr = __popc(eq & lm);
                    h -= p.match * nr + p.mismatch * ((int32_t)run - nr);
                    gapm = __shfl_sync(kFull, gapm, run & 31u);
                    if (run < 32u && h > 0 && gapm) {
                        if (lane == 0 && in_range(k, (uint64_t)m + n, p.err, kSiteLocalMoves)) mv[k] = (uint8_t)gapm;
                        ++k;
                        h -= p.gap;
                        i -= gapm == 1u;
                        j -= gapm == 2u;
                    }
                }
            }
            if (threadIdx.x == 0) {
                if (in_range(tk.out, p.out_cap, p.err, kSiteLocalOut)) {
                    p.ends[4 * (size_t)tk.out + 0] = i;
                    p.ends[4 * (size_t)tk.out + 1] = j;
                }
                nmoves[q] = k;
            }
            __syncthreads();
        }
        __syncwarp();
    }
}

template <int R, int MODE, bool TAB>
int launch_local_R(nw_ctx *ctx, const char *name, LocalArgs &la) {
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_local<R, MODE, TAB>, kLocalWarps * 32, 0);
    if (occ < 1) occ = 1;
    // every CTA resident: a job's warp may wait on an earlier job's warp
    uint32_t blocks = (uint32_t)occ * (uint32_t)ctx->sm_count;
    const uint32_t need = (la.njobs + kLocalWarps - 1) / kLocalWarps;
    if (blocks > need) blocks = need ? need : 1;
    void *v = nullptr;
    int rc = scratch(ctx, "local_counter", 16, &v);
    if (rc) return rc;
    la.counter = (uint32_t *)v;
    cudaMemsetAsync(la.counter, 0, 4, ctx->stream);
    LaunchTimer t(ctx, name);
    k_local<R, MODE, TAB><<<blocks, kLocalWarps * 32, 0, ctx->stream>>>(la);
    return NW_OK;
}

int launch_local(nw_ctx *ctx, int R, LocalMode mode, const char *name, LocalArgs &la) {
    // Scores from shared memory (TAB) take 8 operations a column off the logic pipe
    // and put a shared load into the column's chain: they pay from about three
    // warps per scheduler on.  Pairs of 200 bases and 50 kb, table / permutes: 50 to
    // 1,200 pairs 5.5 / 4.9 ms, 2,400 6.9 / 7.5, 4,800 12.9 / 14.3; 100 pairs of 3 kb
    // (1,200 jobs) .87 / .83, 500 (6,000) 1.47 / 1.71.
    const bool tab = la.njobs > 12u * (uint32_t)ctx->sm_count;
#define NW_LOCAL_CASES(MODEV)                                                      \
    switch (R) {                                                                   \
        case 4: return launch_local_R<4, MODEV, false>(ctx, name, la);             \
        case 16: return launch_local_R<16, MODEV, true>(ctx, name, la);            \
        default: return tab ? launch_local_R<8, MODEV, true>(ctx, name, la)        \
                            : launch_local_R<8, MODEV, false>(ctx, name, la);      \
    }
    if (mode == kKeep) NW_LOCAL_CASES(kKeep)
    if (mode == kEnds) NW_LOCAL_CASES(kEnds)
    NW_LOCAL_CASES(kScore)
#undef NW_LOCAL_CASES
}

template <int R, bool WALK>
int launch_local_trace_R(nw_ctx *ctx, const LocalArgs &la, uint32_t ntasks, uint8_t *moves, const uint64_t *move_off,
                         uint64_t *nmoves) {
    constexpr int smem = WALK ? kTraceWarps * (int)kTileSteps * 32 * (int)sizeof(typename LocalBits<R>::Word) : 0;
    if (smem + 64 > 48 * 1024) {  // (with the static words)
        // one value for every caller: the attribute belongs to the process
        const cudaError_t e =
            cudaFuncSetAttribute(k_local_trace<R, WALK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "local trace shared memory");
    }
    LaunchTimer t(ctx, WALK ? "local_walk" : "local_ends");
    k_local_trace<R, WALK><<<std::min<uint32_t>(ntasks, 65535), WALK ? 32 * kTraceWarps : 32, smem, ctx->stream>>>(
        la, ntasks, moves, move_off, nmoves);
    return NW_OK;
}

template <bool WALK>
int launch_local_trace(nw_ctx *ctx, int R, const LocalArgs &la, uint32_t ntasks, uint8_t *moves,
                       const uint64_t *move_off, uint64_t *nmoves) {
    if (R == 4) return launch_local_trace_R<4, WALK>(ctx, la, ntasks, moves, move_off, nmoves);
    if (R == 16) return launch_local_trace_R<16, WALK>(ctx, la, ntasks, moves, move_off, nmoves);
    return launch_local_trace_R<8, WALK>(ctx, la, ntasks, moves, move_off, nmoves);
}

// (the caller waits for the copy: uploaded)
template <typename T>
int upload_vec(nw_ctx *ctx, const char *slot, const std::vector<T> &v, T **dev) {
    void *d = nullptr;
    int rc = to_device(ctx, v.data(), v.size() * sizeof(T), slot, &d);
    if (rc) return rc;
    *dev = (T *)d;
    return NW_OK;
}

// Waits for the copies of host vectors that the caller is about to free.
int uploaded(nw_ctx *ctx) {
    const cudaError_t e = cudaStreamSynchronize(ctx->stream);
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "task upload sync");
}

// Row profiles of the plain scores s (the global kernels use s - 2*gap).
void local_profile(const nw_scoring &sc, uint32_t prof[4]) {
    for (int c = 0; c < 4; ++c) {
        uint32_t w = 0;
        for (int d = 0; d < 4; ++d) w |= (uint32_t)(uint8_t)(int8_t)(c == d ? sc.match : sc.mismatch) << (8 * d);
        prof[c] = w;
    }
}

int local_device(nw_ctx *ctx, const uint8_t *pool, const uint64_t *a_off, const uint32_t *a_len,
                 const uint64_t *b_off, const uint32_t *b_len, uint32_t npairs, const nw_scoring &sc, uint32_t flags,
                 int32_t *scores, uint32_t *ends, char *cigar_pool, const uint64_t *cigar_off, uint64_t *cigar_len) {
    const bool want = flags & NW_CIGAR;
    int R = 8;
    if (const char *e = getenv("NW_LOCAL_R")) R = atoi(e) == 4 ? 4 : atoi(e) == 16 ? 16 : 8;
    const uint32_t SH = 32u * R;
    LocalMode mode = want ? kKeep : ends ? kEnds : kScore;
    LocalArgs la{};
    la.pool = pool;
    local_profile(sc, la.prof);
    la.match = sc.match;
    la.mismatch = sc.mismatch;
    la.gap = sc.gap;
    la.scores = scores;
    la.ends = ends;
    la.err = ctx->d_err;
    la.out_cap = npairs;
    // Waves that fit a third of the free budget with all they take: stripe rows,
    // kept states, and the moves and tables, which are most of it for short
    // pairs.  A third, because the slots keep the largest size of every wave.
    const uint64_t wave_budget = (ctx->budget - std::min(ctx->budget, ctx->used)) / 3;
    const uint32_t state_units = ((uint32_t)R + 5u) / 4u * 32u;  // 16-byte units of a kept state
    uint64_t kept = 0;
    std::vector<LocalTask> all(npairs);
    for (uint32_t k = 0; k < npairs; ++k) {
        LocalTask &t = all[k];
        t = LocalTask{a_off[k], b_off[k], a_len[k], b_len[k], k, 0, 0, 0, 0, 0};
        // a pair's stripe steps are limited to a 32-bit count
        if ((uint64_t)((t.m + SH - 1) / SH) * std::max(t.n, kLocalMinPeriod) >= (1ull << 31))
            return fail(ctx, NW_ERR_UNSUPPORTED, "pair %u too large for one warp (m*n/%u >= 2^31)", k, SH);
        t.nr = (t.n + 31) / 32 * 32;
        // states before steps kTileSteps, 2 kTileSteps, .. of a stripe's n + 31
        const uint32_t S = (t.m + SH - 1) / SH, states = t.m && t.n ? (t.n + 30) / kTileSteps : 0;
        if (want || (ends && S <= kEndStripes)) t.keep_n = states;
        kept += want ? 0 : (uint64_t)S * t.keep_n * state_units * 16;
    }
    // End cells alone: the states of pairs of few stripes, where they fit.
    if (mode == kEnds && kept > wave_budget / 2)
        for (LocalTask &t : all) t.keep_n = 0;
    else if (mode == kEnds && kept)
        mode = kKeep;
    // longest first (the atomic queue then balances the tail)
    std::vector<uint64_t> cells(npairs);
    for (uint32_t q = 0; q < npairs; ++q) cells[q] = (uint64_t)all[q].m * all[q].n;
    const std::vector<uint32_t> order = radix_order_desc(std::move(cells));
    int rc;
    cudaError_t e0 = cudaMemsetAsync(scores, 0, (size_t)npairs * 4, ctx->stream);  // the stripes' maxima are merged
    if (e0 != cudaSuccess) return cuda_fail(ctx, e0, "local scores reset");
    const bool ends_only = !want && mode != kScore;
    const uint64_t per_job = sizeof(LocalJob) + 4 + (mode == kScore ? 0 : sizeof(LocalBest));
    size_t k0 = 0;
    while (k0 < all.size()) {
        std::vector<LocalTask> wave;
        std::vector<LocalJob> jobs;
        std::vector<uint64_t> moff;
        uint64_t units = 0, rows = 0, mbytes = 0, bytes = 0;
        bool turn = mode == kScore;  // rows: two in turn
        size_t k = k0;
        wave.reserve(all.size() - k0);
        jobs.reserve(all.size() - k0);
        if (want) moff.reserve(all.size() - k0);
        for (; k < all.size(); ++k) {
            LocalTask t = all[order[k]];
            const uint32_t S = (t.m && t.n) ? (t.m + SH - 1) / SH : 1;
            uint64_t u = (uint64_t)S * t.keep_n * state_units;
            uint64_t rw = (uint64_t)(mode == kScore ? std::min(S - 1, 2u) : S - 1) * t.nr;
            const uint64_t tables = sizeof(LocalTask) + S * per_job +
                                    (want ? t.m + t.n + 16 + 2 * sizeof(uint64_t) + sizeof(TraceTask) : 0);
            const uint64_t more = u * 16 + rw * 4 + tables;
            if (!wave.empty() && ((turn && ends_only) || bytes + more > wave_budget)) break;
            bytes += more;
            // a lone pair whose rows alone exceed the budget keeps two and
            // finds its end cell by sweeping the stripes above it again
            if (ends_only && wave.empty() && rw * 4 + tables + (64u << 10) > scratch_headroom(ctx, "local_rows")) {
                turn = true;
                rw = (uint64_t)std::min(S - 1, 2u) * t.nr;
                t.keep_n = 0;  // (a replay from a state reads the row above, which may be overwritten)
                u = 0;
            }
            t.keep_off = units;
            t.row_off = rows;
            t.job0 = (uint32_t)jobs.size();
            for (uint32_t s = 0; s < S; ++s) jobs.push_back(LocalJob{(uint32_t)wave.size(), s});
            units += u;
            rows += rw;
            if (want) moff.push_back(mbytes);
            mbytes += (uint64_t)t.m + t.n + 16;
            wave.push_back(t);
        }
        void *kv = nullptr, *rv = nullptr, *pv = nullptr, *bv = nullptr, *mv = nullptr, *nm = nullptr;
        if ((rc = scratch(ctx, "local_rows", rows * 4 + 16, &rv))) return rc;
        if ((rc = scratch(ctx, "local_progress", jobs.size() * 4 + 16, &pv))) return rc;
        if (mode != kScore && (rc = scratch(ctx, "local_best", jobs.size() * sizeof(LocalBest) + 16, &bv))) return rc;
        if (mode == kKeep && (rc = scratch(ctx, "local_keep", units * 16 + 16, &kv))) return rc;
        if (want) {
            if ((rc = scratch(ctx, "local_moves", mbytes + 16, &mv))) return rc;
            if ((rc = scratch(ctx, "local_nmoves", wave.size() * 8 + 16, &nm))) return rc;
        }
        if ((e0 = cudaMemsetAsync(pv, 0, jobs.size() * 4, ctx->stream)) != cudaSuccess)
            return cuda_fail(ctx, e0, "local progress reset");
        // A fill that gives up (a wait's limit, or an error that the context
        // holds from an earlier call) leaves jobs undone.  Their best reads 0,
        // so the trace starts only from stripes that were finished -- and then
        // every stripe above them was: a stripe reads all of the one above.
        if (mode != kScore && (e0 = cudaMemsetAsync(bv, 0, jobs.size() * sizeof(LocalBest), ctx->stream)) != cudaSuccess)
            return cuda_fail(ctx, e0, "local best reset");
        LocalTask *dt = nullptr;
        LocalJob *dj = nullptr;
        uint64_t *dmoff = nullptr;
        if ((rc = upload_vec(ctx, "local_tasks", wave, &dt))) return rc;
        if ((rc = upload_vec(ctx, "local_jobs", jobs, &dj))) return rc;
        if (want && (rc = upload_vec(ctx, "local_move_off", moff, &dmoff))) return rc;
        if ((rc = uploaded(ctx))) return rc;
        la.tasks = dt;
        la.jobs = dj;
        la.njobs = (uint32_t)jobs.size();
        la.rows = (uint32_t *)rv;
        la.rows_cap = rows;
        la.turn = turn;
        la.progress = (uint32_t *)pv;
        la.best = (LocalBest *)bv;
        la.keep = (uint4 *)kv;
        la.keep_cap = units;
        const uint32_t nt = (uint32_t)wave.size();
        k0 = k;
        if ((rc = launch_local(ctx, R, mode, want ? "local_fill_ptr" : ends_only ? "local_score_pos" : "local_score", la)))
            return rc;
        if (ends_only && (rc = launch_local_trace<false>(ctx, R, la, nt, nullptr, nullptr, nullptr))) return rc;
        if (!want) continue;
        if ((rc = launch_local_trace<true>(ctx, R, la, nt, (uint8_t *)mv, dmoff, (uint64_t *)nm))) return rc;
        std::vector<TraceTask> tt(wave.size());
        for (size_t q = 0; q < wave.size(); ++q) {
            const LocalTask &t = wave[q];
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
            x.origin = ends + 4 * (size_t)t.out;
            tt[q] = x;
        }
        TraceTask *dtt = nullptr;
        if ((rc = upload_vec(ctx, "local_trace_tasks", tt, &dtt)) || (rc = uploaded(ctx))) return rc;
        if ((rc = launch_finish(ctx, tt[0], dtt, (uint32_t)tt.size(), (flags & NW_CIGAR_M) ? 1u : 0u))) return rc;
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "local launch");
}

uint64_t pool_extent(const uint64_t *a_off, const uint32_t *a_len, const uint64_t *b_off, const uint32_t *b_len,
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

extern "C" int nw_local_align_batch(nw_ctx *ctx, const uint8_t *pool2b, const uint64_t *a_off, const uint32_t *a_len,
                                    const uint64_t *b_off, const uint32_t *b_len, uint32_t npairs, nw_scoring sc,
                                    uint32_t flags, int32_t *scores, uint32_t *ends, char *cigar_pool,
                                    const uint64_t *cigar_off, uint64_t *cigar_len) {
    if (!ctx) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    int rc = check_scoring(ctx, sc);
    if (rc) return rc;
    if (npairs == 0) return NW_OK;
    const bool want = flags & NW_CIGAR;
    if (!pool2b || !a_off || !a_len || !b_off || !b_len || !scores) return fail(ctx, NW_ERR_ARG, "null argument");
    if (want && (!ends || !cigar_pool || !cigar_off || !cigar_len))
        return fail(ctx, NW_ERR_ARG, "NW_CIGAR needs ends and CIGAR buffers");
    for (uint32_t k = 0; k < npairs; ++k) {
        if (a_len[k] >= (1u << 30) || b_len[k] >= (1u << 30)) return fail(ctx, NW_ERR_ARG, "sequence longer than 2^30");
        const uint64_t mn = std::min(a_len[k], b_len[k]);
        if ((uint64_t)std::max(sc.match, 0) * mn >= (1ull << 29))
            return fail(ctx, NW_ERR_ARG, "match * min(m,n) must stay below 2^29");
        if (want && cigar_off[k + 1] - cigar_off[k] < nw_cigar_bound(a_len[k], b_len[k]))
            return fail(ctx, NW_ERR_ARG, "CIGAR capacity of pair %u below nw_cigar_bound", k);
    }
    if (!(flags & NW_HOST_IO))
        return local_device(ctx, pool2b, a_off, a_len, b_off, b_len, npairs, sc, flags, scores, ends, cigar_pool,
                            cigar_off, cigar_len);
    void *dp = nullptr, *ds = nullptr, *de = nullptr, *dc = nullptr, *dl = nullptr;
    if ((rc = to_device(ctx, pool2b, pool_extent(a_off, a_len, b_off, b_len, npairs), "hio_pool", &dp))) return rc;
    if ((rc = scratch(ctx, "hio_scores", (size_t)npairs * 4, &ds))) return rc;
    if (ends && (rc = scratch(ctx, "hio_ends", (size_t)npairs * 16, &de))) return rc;
    if (want) {
        if ((rc = scratch(ctx, "hio_cigar", cigar_off[npairs] + 16, &dc))) return rc;
        if ((rc = scratch(ctx, "hio_cigar_len", (size_t)npairs * 8, &dl))) return rc;
    }
    if ((rc = local_device(ctx, (const uint8_t *)dp, a_off, a_len, b_off, b_len, npairs, sc, flags, (int32_t *)ds,
                           (uint32_t *)de, (char *)dc, cigar_off, (uint64_t *)dl)))
        return rc;
    cudaError_t e = cudaMemcpyAsync(scores, ds, (size_t)npairs * 4, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && ends) e = cudaMemcpyAsync(ends, de, (size_t)npairs * 16, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && want) e = cudaMemcpyAsync(cigar_len, dl, (size_t)npairs * 8, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && want)
        e = cudaMemcpyAsync(cigar_pool, dc, cigar_off[npairs], cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "local D2H");
    return nw_ctx_sync(ctx);
}
