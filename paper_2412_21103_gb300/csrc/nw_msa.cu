// Center-star multiple alignment (the paper's Sec. 3.2) on one GPU.
//
// Stage 1, the scoring matrix: the n(n-1)/2 pairwise scores of Eq. 2 by the
// batched kernel (nw_score_all_pairs).  Stage 2, the center: the sequence
// most similar to the rest -- the largest sum of its scores against the
// other sequences (the diagonal len*match is left out), lowest index on
// ties -- found by a row-sum kernel and an arg-max kernel.  Stage 3: every
// sequence aligned (as the query, rows) with the center (the reference,
// columns) by the batched CIGAR path.  Stage 4, the merge with the aligned
// center as the reference ("once a gap, always a gap"): before center base
// p (p = 0..|C|, |C| = after the last base) the merged alignment keeps G[p]
// columns, the most 'I' ops any alignment puts there; center base p lands in
// column p + G[0] + ... + G[p]; a row's I-bases fill their slot from its
// left; a 'D' op leaves '-' in the center's column.  The merge reads the
// RLE CIGARs on the device: one warp per sequence finds its insertion
// runs (atomic max into G), one block scans G into column offsets, one
// warp per sequence writes its row.
#include <algorithm>
#include <vector>

#include "nw_internal.cuh"

namespace nw {

// Sum of row i over j != i (int64), one warp per row.
__global__ void k_row_sums(const int32_t *M, uint32_t nseq, int64_t *sums) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nseq; i += warps) {
        const int32_t *row = M + (size_t)i * nseq;
        int64_t s = 0;
        for (uint32_t j = lane; j < nseq; j += 32u)
            if (j != i) s += row[j];
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (lane == 0) sums[i] = s;
    }
}

// Index of the largest sum, the lowest index on ties (one block).
__global__ void k_argmax(const int64_t *sums, uint32_t nseq, uint32_t *center) {
    __shared__ int64_t bv[32];
    __shared__ uint32_t bi[32];
    int64_t v = INT64_MIN;
    uint32_t idx = 0xffffffffu;
    for (uint32_t i = threadIdx.x; i < nseq; i += blockDim.x)
        if (sums[i] > v) {  // i grows: strict keeps the first maximum of this thread
            v = sums[i];
            idx = i;
        }
    auto better = [](int64_t v1, uint32_t i1, int64_t v2, uint32_t i2) { return v1 > v2 || (v1 == v2 && i1 < i2); };
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const int64_t v2 = __shfl_xor_sync(kFull, v, o);
        const uint32_t i2 = __shfl_xor_sync(kFull, idx, o);
        if (better(v2, i2, v, idx)) {
            v = v2;
            idx = i2;
        }
    }
    const uint32_t w = threadIdx.x >> 5, nw_ = (blockDim.x + 31) >> 5;
    if ((threadIdx.x & 31u) == 0) {
        bv[w] = v;
        bi[w] = idx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (uint32_t k = 1; k < nw_; ++k)
            if (better(bv[k], bi[k], v, idx)) {
                v = bv[k];
                idx = bi[k];
            }
        *center = idx;
    }
}

// The runs of a CIGAR, 32 characters at a time: f(op, ch, cnt) gets whether the
// lane's character is an operation, which, and its count (valid where it is
// one), by the whole warp; ends early, false, when f does or a character is none
// of a CIGAR's.  A number is put together by a scan over the characters (value
// and power of ten), the digits left over from the characters before carried
// along.  A warp's lanes take the runs side by side: one after another, the
// merge of 512 sequences of 500 to 1,500 bases took .21 and .23 ms
// (gaps, rows), now .05 and .06.
template <typename F>
__device__ bool for_runs(const char *c, uint64_t len, uint32_t lane, F f) {
    uint64_t open = 0;  // the number that the characters before end with
    for (uint64_t q0 = 0; q0 < len; q0 += 32) {
        const bool in = q0 + lane < len;
        const char ch = in ? c[q0 + lane] : '=';
        const bool digit = ch >= '0' && ch <= '9';
        const bool op = in && (ch == '=' || ch == 'X' || ch == 'M' || ch == 'I' || ch == 'D');
        // the number of the digits up to and with this lane: v digits-to-here, p its power of ten
        uint64_t v = digit ? (uint64_t)(ch - '0') : 0u, p = digit ? 10u : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t v2 = __shfl_up_sync(kFull, v, o), p2 = __shfl_up_sync(kFull, p, o);
            if ((int)lane >= o) {
                v += p * v2;  // p is 0 once a lane that is no digit lies between
                p *= p2;
            }
        }
        v += p * open;  // digits from the first character on continue the open number
        const uint32_t last = (uint32_t)min((unsigned long long)(len - q0), 32ull) - 1u;
        const uint64_t before = __shfl_up_sync(kFull, v, 1);
        const uint64_t cnt = lane ? before : open;
        open = __shfl_sync(kFull, v, last);
        if (!f(op, ch, cnt) || __any_sync(kFull, in && !digit && !op)) return false;
    }
    return true;
}

template <typename T>
__device__ __forceinline__ T warp_incl(T v, uint32_t lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(kFull, v, o);
        if ((int)lane >= o) v += y;
    }
    return v;
}

// Where 32 characters' runs stand, from the center bases p and the bases i used
// before them and the insertions `ins` that the characters before end with.
// EMPTY: a run of no bases ends them too.
template <typename T, bool EMPTY>
struct RunPlaces {
    T dp, di, p0, i1, p1, i_off;  // consumed by the run; before it (p) and after it (i, p); bases of the chunk with it
    T ins;                        // insertions right before it
    __device__ RunPlaces(bool op, char ch, T cnt, uint32_t lane, T &p, T &i, T &carry) {
        const bool is_i = op && ch == 'I';
        dp = op && !is_i ? cnt : T(0);
        di = op && ch != 'D' ? cnt : T(0);
        const T P = warp_incl(dp, lane), Q = warp_incl(di, lane), d = is_i ? cnt : T(0), N = warp_incl(d, lane);
        p1 = p + P;
        p0 = p1 - dp;
        i_off = Q;
        i1 = i + Q;
        // a run that is no insertion ends the ones before it
        const uint32_t ends = __ballot_sync(kFull, op && !is_i && (EMPTY || cnt)), before = ends & ((1u << lane) - 1u);
        const T N_end = __shfl_sync(kFull, N, before ? 31 - __clz(before) : 0);
        ins = N - d - (before ? N_end : T(0)) + (before ? T(0) : carry);
        const T N_all = __shfl_sync(kFull, N, 31), N_last = __shfl_sync(kFull, N, ends ? 31 - __clz(ends) : 0);
        carry = ends ? N_all - N_last : carry + N_all;
        p += __shfl_sync(kFull, P, 31);
        i += __shfl_sync(kFull, Q, 31);
    }
};

// G[p] = max over sequences of the 'I' ops placed before center base p.
// Checks that alignment k consumes exactly len[k] bases and the C center
// bases (NW_ERR_ARG into the error word, detail k, otherwise).
__global__ void k_slot_gaps(const char *cigar_pool, const uint64_t *cigar_off, const uint64_t *cigar_len,
                            const uint32_t *len, uint32_t nseq, uint32_t C, uint32_t *G, uint32_t *err) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < nseq; k += (gridDim.x * blockDim.x) >> 5) {
        uint64_t p = 0, i = 0, ins = 0;
        auto slot = [&](uint64_t at, uint64_t n) {
            if (n && at <= C) atomicMax(G + at, n < 0xffffffffull ? (uint32_t)n : 0xffffffffu);
        };
        const bool ok = for_runs(cigar_pool + cigar_off[k], cigar_len[k], lane, [&](bool op, char ch, uint64_t cnt) {
            const RunPlaces<uint64_t, true> r(op, ch, cnt, lane, p, i, ins);
            if (__any_sync(kFull, op && (r.p1 > C || r.i1 > len[k]))) return false;
            if (op && ch != 'I') slot(r.p0, r.ins);
            return true;
        });
        if (lane == 0) {
            slot(p, ins);
            if (!ok || p != C || i != len[k]) raise_error(err, NW_ERR_ARG, k);
        }
    }
}

// start[p] = p + G[0] + ... + G[p-1] (first column of slot p) for p =
// 0..count-1, and the column count (count-1) + sum(G) (one block).
__global__ void k_slot_scan(const uint32_t *G, uint32_t count, uint64_t *start, uint64_t *ncols) {
    __shared__ uint64_t wsum[32];
    __shared__ uint64_t carry_s;
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (uint32_t base = 0; base < count; base += blockDim.x) {
        const uint32_t p = base + threadIdx.x;
        const uint64_t v = p < count ? (uint64_t)G[p] : 0u;
        uint64_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(kFull, incl, o);
            if ((int)lane >= o) incl += y;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        if (w == 0) {
            uint64_t t = lane < nwarps ? wsum[lane] : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t y = __shfl_up_sync(kFull, t, o);
                if ((int)lane >= o) t += y;
            }
            if (lane < nwarps) wsum[lane] = t;  // inclusive over warps
        }
        __syncthreads();
        const uint64_t before = carry_s + (w ? wsum[w - 1] : 0u) + (incl - v);
        if (p < count) start[p] = before + p;
        __syncthreads();
        if (threadIdx.x == 0) carry_s += wsum[nwarps - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) *ncols = carry_s + (count - 1);
}

// Row k of the merged alignment: the caller set every byte to '-'.
__global__ void k_merge_rows(const uint8_t *pool, const uint64_t *off, const uint32_t *len, const char *cigar_pool,
                             const uint64_t *cigar_off, const uint64_t *cigar_len, uint32_t nseq, const uint32_t *G,
                             const uint64_t *start, const uint64_t *ncols, char *msa, uint64_t ld,
                             uint32_t *err) {
    if (*(volatile const uint32_t *)err) return;  // a CIGAR failed its check
    const uint64_t cols = *ncols;
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < nseq; k += (gridDim.x * blockDim.x) >> 5) {
        char *row = msa + (uint64_t)k * ld;
        const uint8_t *s = pool + off[k];
        uint32_t p = 0, i = 0, used = 0;  // the CIGAR passed its check: all within 32 bits
        for_runs(cigar_pool + cigar_off[k], cigar_len[k], lane, [&](bool op, char ch, uint64_t cnt) {
            const uint32_t i0 = i;
            const RunPlaces<uint32_t, false> r(op, ch, (uint32_t)cnt, lane, p, i, used);
            // the chunk's bases by the lanes, each from the first run that reaches it
            const uint32_t bases = i - i0;
            for (uint32_t b0 = 0; b0 < bases; b0 += 32) {
                const uint32_t b = b0 + lane;
                uint32_t at = 0;
#pragma unroll
                for (uint32_t o = 16; o; o >>= 1)
                    if (__shfl_sync(kFull, r.i_off, at + o - 1) <= b) at += o;
                at = min(at, 31u);
                const uint32_t x = b - (__shfl_sync(kFull, r.i_off, at) - __shfl_sync(kFull, r.di, at));  // within the run
                const uint32_t p0 = __shfl_sync(kFull, r.p0, at), ins = __shfl_sync(kFull, r.ins, at);
                const bool is_i = __shfl_sync(kFull, (int)ch, at) == 'I';
                if (b < bases) {
                    const uint64_t col = is_i ? start[p0] + ins + x : start[p0 + x] + G[p0 + x];
                    if (in_range(col, cols, err, kSiteMsaRow)) row[col] = "ACGT"[base_at(s, i0 + b)];
                }
            }
            return true;
        });
        if (lane == 0 && ld > cols) row[cols] = '\0';
    }
}

// The merge on device buffers (metadata arrays on the host).
static int merge_device(nw_ctx *ctx, const uint8_t *pool, const uint64_t *off, const uint32_t *len, uint32_t nseq,
                        uint32_t center, const char *cigar_pool, const uint64_t *cigar_off, const uint64_t *cigar_len,
                        char *msa, uint64_t ld, uint64_t *msa_cols) {
    int rc;
    const uint32_t C = len[center];
    void *doff = nullptr, *dlen = nullptr, *dcoff = nullptr, *dG = nullptr, *dstart = nullptr, *dn = nullptr;
    if ((rc = to_device(ctx, off, (size_t)nseq * 8, "msa_off", &doff))) return rc;
    if ((rc = to_device(ctx, len, (size_t)nseq * 4, "msa_len", &dlen))) return rc;
    if ((rc = to_device(ctx, cigar_off, (size_t)nseq * 8, "msa_coff", &dcoff))) return rc;
    if ((rc = scratch(ctx, "msa_G", ((size_t)C + 1) * 4, &dG))) return rc;
    if ((rc = scratch(ctx, "msa_start", ((size_t)C + 1) * 8, &dstart))) return rc;
    if ((rc = scratch(ctx, "msa_ncols", 16, &dn))) return rc;
    cudaError_t e = cudaMemsetAsync(dG, 0, ((size_t)C + 1) * 4, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "msa memset");
    const uint32_t blocks = std::max<uint32_t>(1, (nseq + 3) / 4);  // a warp per sequence
    {
        LaunchTimer t(ctx, "msa_gaps");
        k_slot_gaps<<<blocks, 128, 0, ctx->stream>>>(cigar_pool, (const uint64_t *)dcoff, cigar_len,
                                                     (const uint32_t *)dlen, nseq, C, (uint32_t *)dG, ctx->d_err);
    }
    {
        LaunchTimer t(ctx, "msa_scan");
        k_slot_scan<<<1, 1024, 0, ctx->stream>>>((const uint32_t *)dG, C + 1, (uint64_t *)dstart, (uint64_t *)dn);
    }
    uint64_t cols = 0;
    e = cudaMemcpyAsync(&cols, dn, 8, cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "msa column count D2H");
    if ((rc = nw_ctx_sync(ctx))) return rc;
    *msa_cols = cols;
    if (!msa) return NW_OK;
    if (ld < cols) return fail(ctx, NW_ERR_CIGAR_TRUNC, "merged alignment has %llu columns, row stride is %llu",
                               (unsigned long long)cols, (unsigned long long)ld);
    if (nseq && (e = cudaMemsetAsync(msa, '-', (size_t)nseq * ld, ctx->stream)) != cudaSuccess)
        return cuda_fail(ctx, e, "msa fill");
    {
        LaunchTimer t(ctx, "msa_rows");
        k_merge_rows<<<blocks, 128, 0, ctx->stream>>>(pool, (const uint64_t *)doff, (const uint32_t *)dlen,
                                                      cigar_pool, (const uint64_t *)dcoff, cigar_len, nseq,
                                                      (const uint32_t *)dG, (const uint64_t *)dstart,
                                                      (const uint64_t *)dn, msa, ld, ctx->d_err);
    }
    e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "msa launch");
}

static uint64_t pool_extent(const uint64_t *off, const uint32_t *len, uint32_t nseq) {
    uint64_t b = 16;
    for (uint32_t k = 0; k < nseq; ++k) b = std::max<uint64_t>(b, off[k] + (len[k] + 3) / 4);
    return b;
}

}  // namespace nw

using namespace nw;

extern "C" int nw_msa_merge(nw_ctx *ctx, const uint8_t *pool2b, const uint64_t *off, const uint32_t *len,
                            uint32_t nseq, uint32_t center, uint32_t flags, const char *cigar_pool,
                            const uint64_t *cigar_off, const uint64_t *cigar_len, char *msa, uint64_t msa_ld,
                            uint64_t *msa_cols) {
    if (!ctx) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    if (nseq == 0) return fail(ctx, NW_ERR_ARG, "no sequences");
    if (!pool2b || !off || !len || !cigar_pool || !cigar_off || !cigar_len || !msa_cols || center >= nseq)
        return fail(ctx, NW_ERR_ARG, "null argument or center out of range");
    if (!(flags & NW_HOST_IO))
        return merge_device(ctx, pool2b, off, len, nseq, center, cigar_pool, cigar_off, cigar_len, msa, msa_ld,
                            msa_cols);
    int rc;
    void *dp = nullptr, *dc = nullptr, *dl = nullptr, *dm = nullptr;
    if ((rc = to_device(ctx, pool2b, pool_extent(off, len, nseq), "hio_pool", &dp))) return rc;
    uint64_t extent = 16;
    for (uint32_t k = 0; k < nseq; ++k) extent = std::max<uint64_t>(extent, cigar_off[k] + cigar_len[k]);
    if ((rc = to_device(ctx, cigar_pool, extent, "hio_cigar", &dc))) return rc;
    if ((rc = to_device(ctx, cigar_len, (size_t)nseq * 8, "hio_cigar_len", &dl))) return rc;
    if (msa && (rc = scratch(ctx, "hio_msa", (size_t)nseq * msa_ld + 16, &dm))) return rc;
    if ((rc = merge_device(ctx, (const uint8_t *)dp, off, len, nseq, center, (const char *)dc, cigar_off,
                           (const uint64_t *)dl, msa ? (char *)dm : nullptr, msa_ld, msa_cols)))
        return rc;
    if (!msa) return NW_OK;
    cudaError_t e = cudaMemcpyAsync(msa, dm, (size_t)nseq * msa_ld, cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "msa D2H");
    return nw_ctx_sync(ctx);
}

extern "C" int nw_center_star(nw_ctx *ctx, const uint8_t *pool2b, const uint64_t *off, const uint32_t *len,
                              uint32_t nseq, nw_scoring sc, uint32_t flags, uint32_t *center, int64_t *row_sums,
                              int32_t *scores, char *cigar_pool, const uint64_t *cigar_off, uint64_t *cigar_len,
                              char *msa, uint64_t msa_ld, uint64_t *msa_cols) {
    if (!ctx) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    int rc = check_scoring(ctx, sc);
    if (rc) return rc;
    if (nseq == 0 || nseq > 65535) return fail(ctx, NW_ERR_ARG, "1 to 65535 sequences");
    if (!pool2b || !off || !len || !center || !scores || !cigar_pool || !cigar_off || !cigar_len || !msa_cols)
        return fail(ctx, NW_ERR_ARG, "null argument");
    for (uint32_t k = 0; k < nseq; ++k)
        if (cigar_off[k + 1] < cigar_off[k]) return fail(ctx, NW_ERR_ARG, "CIGAR offsets must not decrease");
    const bool host = flags & NW_HOST_IO;
    const uint8_t *pool = pool2b;
    int32_t *d_scores = scores;
    char *d_cig = cigar_pool;
    uint64_t *d_clen = cigar_len;
    int64_t *d_sums = row_sums;
    if (host) {
        void *p = nullptr;
        if ((rc = to_device(ctx, pool2b, pool_extent(off, len, nseq), "hio_pool", &p))) return rc;
        pool = (const uint8_t *)p;
        if ((rc = scratch(ctx, "hio_scores", (size_t)nseq * 4, &p))) return rc;
        d_scores = (int32_t *)p;
        if ((rc = scratch(ctx, "hio_cigar", cigar_off[nseq] + 16, &p))) return rc;
        d_cig = (char *)p;
        if ((rc = scratch(ctx, "hio_cigar_len", (size_t)nseq * 8, &p))) return rc;
        d_clen = (uint64_t *)p;
        d_sums = nullptr;
    }
    // stage 1: the scoring matrix (Eq. 2 pairs)
    void *dM = nullptr, *dS = nullptr, *dc = nullptr;
    cudaError_t e0 = cudaSuccess;
    if ((rc = scratch(ctx, "cs_matrix", (size_t)nseq * nseq * 4, &dM))) return rc;
    if (!d_sums) {
        if ((rc = scratch(ctx, "cs_sums", (size_t)nseq * 8, &dS))) return rc;
        d_sums = (int64_t *)dS;
    }
    if ((rc = scratch(ctx, "cs_center", 16, &dc))) return rc;
    if (nseq == 1) {  // no pair to score: the one sequence is the center
        if ((e0 = cudaMemsetAsync(dM, 0, 4, ctx->stream)) != cudaSuccess) return cuda_fail(ctx, e0, "matrix");
    } else if ((rc = nw_score_all_pairs(ctx, pool, off, len, nseq, sc, flags & NW_GRAPH, (int32_t *)dM))) {
        return rc;
    }
    // stage 2: the center
    {
        LaunchTimer t(ctx, "center", 2);
        const uint32_t blocks = std::min<uint32_t>((nseq + 7) / 8, (uint32_t)ctx->sm_count * 8);
        k_row_sums<<<blocks, 256, 0, ctx->stream>>>((const int32_t *)dM, nseq, d_sums);
        k_argmax<<<1, 1024, 0, ctx->stream>>>(d_sums, nseq, (uint32_t *)dc);
    }
    uint32_t c = 0;
    cudaError_t e = cudaMemcpyAsync(&c, dc, 4, cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "center D2H");
    if ((rc = nw_ctx_sync(ctx))) return rc;
    *center = c;
    // stage 3: every sequence (query) against the center (reference)
    std::vector<uint64_t> b_off(nseq, off[c]);
    std::vector<uint32_t> b_len(nseq, len[c]);
    for (uint32_t k = 0; k < nseq; ++k)
        if (cigar_off[k + 1] - cigar_off[k] < nw_cigar_bound(len[k], len[c]))
            return fail(ctx, NW_ERR_ARG, "CIGAR capacity of sequence %u below nw_cigar_bound", k);
    if ((rc = nw_align_batch(ctx, pool, off, len, b_off.data(), b_len.data(), nseq, sc,
                             NW_CIGAR | (flags & NW_CIGAR_M), d_scores, d_cig, cigar_off, d_clen)))
        return rc;
    // stage 4: the merge
    char *d_msa = msa;
    if (host && msa) {
        void *p = nullptr;
        if ((rc = scratch(ctx, "hio_msa", (size_t)nseq * msa_ld + 16, &p))) return rc;
        d_msa = (char *)p;
    }
    if ((rc = merge_device(ctx, pool, off, len, nseq, c, d_cig, cigar_off, d_clen, d_msa, msa_ld, msa_cols)))
        return rc;
    if (!host) return NW_OK;
    e = cudaMemcpyAsync(scores, d_scores, (size_t)nseq * 4, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(cigar_len, d_clen, (size_t)nseq * 8, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(cigar_pool, d_cig, cigar_off[nseq], cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && row_sums)
        e = cudaMemcpyAsync(row_sums, d_sums, (size_t)nseq * 8, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && msa) e = cudaMemcpyAsync(msa, d_msa, (size_t)nseq * msa_ld, cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "center-star D2H");
    return nw_ctx_sync(ctx);
}
