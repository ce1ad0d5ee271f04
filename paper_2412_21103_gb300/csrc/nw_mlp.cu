// Learned band (a9): 4-mer diagonal-histogram features and a small BF16 MLP
// that predicts the band half-width of a pair.  Not in the paper.
//
// Features of a pair (A: m bases, B: n bases, L = max(m,n), delta = n - m):
//   K = min(256, m-3) anchors i_k = floor(k*(m-4)/(K-1)) in A; anchor i's
//   expected diagonal is e(i) = round(delta*i/m); every j in B within
//   W = max(1, L/8) of i + e(i) whose 4-mer equals A's 4-mer at i adds one to
//   bin floor((j - i - e(i) + W) * 64 / (2W+1)).  f[b] = log1p(count_b) /
//   log1p(K) for the 64 bins, f[64] = delta / L.  (Pairs with m < 4 or n < 4
//   get an all-zero histogram.)
//
// Network: 65 -> 128 (ReLU) -> 128 (ReLU) -> 1, weights and activations in
// BF16, accumulation and biases in FP32; the output is log(w) of the band
// half-width.  Parameters (FP32 masters, flat): W1[128][65], b1[128],
// W2[128][128], b2[128], W3[128], b3.  Loss: 0.5 * mean((y - t)^2).  Training
// uses Adam (beta 0.9 / 0.999, eps 1e-8) on the FP32 masters; the BF16
// copies used by forward and backward are refreshed after every step.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

#include "nw_internal.cuh"

namespace nw {

constexpr int kF = 65, kH = 128;
constexpr int kNW1 = kH * kF, kNB1 = kH, kNW2 = kH * kH, kNB2 = kH, kNW3 = kH, kNB3 = 1;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kNW1, kOffW2 = kOffB1 + kNB1, kOffB2 = kOffW2 + kNW2,
              kOffW3 = kOffB2 + kNB2, kOffB3 = kOffW3 + kNW3, kNParams = kOffB3 + kNB3;
constexpr int kAnchors = 256, kBins = 64;
constexpr int kShortWindow = 256;  // offsets of a window whose matches are counted one by one (k_features)

struct BandModel {
    float *master = nullptr;      // kNParams
    __nv_bfloat16 *wb = nullptr;  // BF16 copies of W1, W2, W3 (same offsets)
    float *adam_m = nullptr, *adam_v = nullptr;
    float *grad = nullptr;        // kNParams + 1 (gradients and loss)
    int64_t step = 0;
};

// ---------------------------------------------------------------- features
// One CTA per pair, thread k = anchor k, bits instead of codes: B sits in shared
// memory as two bit planes, and a thread's match word, 32 positions of B at
// once, is the AND of its four letters' equality words, the last three shifted
// by 1, 2, 3 (about 25 ALU instructions a word, which bounds the kernel).  A
// thread walks its window of B from offset d = 0, d = j - i - e(i) + W, so every
// lane is at the same d: a bin is the same bit range of the same words in all
// of them, its count a population count and one warp-wide sum, with no atomics
// and no division per match.
//
// The flush of the 64 bins takes about as long as 8 words with a match at every
// position, so a window of up to kShortWindow offsets (sequences under 1,024
// bases) takes its matches one by one: 100,000 pairs of 50 to 150 bases .50 ms, with
// the flush 1.52; byte by byte .47.
//
// One byte per position, compared four at a time, the matches taken out one by
// one with a 64-bit division each and added by atomics: 2.37 ms for 10,000
// pairs of 2 to 20 kb; this form 0.53 ms.
__device__ __forceinline__ void letter_words(const uint2 v, const uint32_t (&c0)[4], const uint32_t (&c1)[4],
                                             uint32_t (&E)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) E[k] = ~((v.x ^ c0[k]) | (v.y ^ c1[k]));
}

template <int CTAS>
__global__ void __launch_bounds__(kAnchors, CTAS) k_features(const uint8_t *pool, const uint64_t *a_off,
                                                       const uint32_t *a_len, const uint64_t *b_off,
                                                       const uint32_t *b_len, uint32_t npairs, float *feat) {
    extern __shared__ uint2 bpl[];  // the bit planes of B, 32 bases an element
    __shared__ uint32_t hist[kBins];
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t p = blockIdx.x; p < npairs; p += gridDim.x) {
        const uint32_t m = a_len[p], n = b_len[p];
        const uint8_t *A = pool + a_off[p], *B = pool + b_off[p];
        if (threadIdx.x < kBins) hist[threadIdx.x] = 0;
        const bool ok = m >= 4 && n >= 4;
        const int32_t nk = ok ? (int32_t)n - 3 : 0, nwords = ok ? (int32_t)((n + 31) / 32) : 0;
        const uint32_t nbytes = (n + 3) / 4;
        for (int32_t w = threadIdx.x; w < nwords; w += kAnchors) {
            uint64_t v = 0;
            const uint32_t at = 8u * (uint32_t)w;
            if (at + 8 <= nbytes) {
#pragma unroll
                for (int k = 0; k < 8; ++k) v |= (uint64_t)B[at + k] << (8 * k);
            } else {
                for (uint32_t k = 0; at + k < nbytes; ++k) v |= (uint64_t)B[at + k] << (8 * k);
            }
            bpl[w] = make_uint2(even_bits(v), even_bits(v >> 1));
        }
        __syncthreads();
        const uint32_t L = max(m, n);
        const int32_t delta = (int32_t)n - (int32_t)m;
        const uint32_t K = ok ? min((uint32_t)kAnchors, m - 3) : 0;
        if ((threadIdx.x & ~31u) < K) {  // a warp with an anchor
            const bool live = threadIdx.x < K;
            uint32_t i = 0;  // (in 32 bits where it fits: the division takes a third of the instructions)
            if (live && K > 1)
                i = m < (1u << 24) ? threadIdx.x * (m - 4) / (K - 1) : (uint32_t)(((uint64_t)threadIdx.x * (m - 4)) / (K - 1));
            uint32_t c0[4], c1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t c = base_at(A, i + k);
                c0[k] = 0u - (c & 1u);
                c1[k] = 0u - (c >> 1);
            }
            const int32_t e = (int32_t)llrint((double)delta * (double)i / (double)m);
            const int32_t W = max(1, (int32_t)(L / 8));
            const int32_t j0 = (int32_t)i + e - W;  // the position at d = 0
            // words of d that hold a position of B for some lane
            const int32_t dlo = __reduce_min_sync(~0u, live ? max(0, -j0) : 0x7FFFFFFF);
            const int32_t dhi = __reduce_max_sync(~0u, live ? min(2 * W, nk - 1 - j0) : -1);
            const int32_t nfull = live ? nk >> 5 : 0;  // words of B whose every position counts
            const uint32_t tail = live ? (1u << (nk & 31)) - 1u : 0u;
            const uint32_t s = (uint32_t)j0 & 31u;
            int32_t t = dlo >> 5;
            int32_t w = (j0 >> 5) + t;  // floor: B's word at the low end of the window
            const auto planes = [&](int32_t q) { return bpl[min(max(q, 0), nwords - 1)]; };
            // match word of B's word q from its letters' words E and the next word's F
            const auto match = [&](int32_t q, const uint32_t (&E)[4], const uint32_t (&F)[4]) {
                uint32_t valid = ~0u;
                if ((uint32_t)q >= (uint32_t)nfull) valid = q == nfull ? tail : 0u;
                return E[0] & __funnelshift_r(E[1], F[1], 1) & __funnelshift_r(E[2], F[2], 2) &
                       __funnelshift_r(E[3], F[3], 3) & valid;
            };
            // f(t, x): the match bits of offsets 32 t .. 32 t + 31
            const auto words = [&](auto f) {
                uint32_t E[4], F[4];
                letter_words(planes(w), c0, c1, E);
                letter_words(planes(w + 1), c0, c1, F);
                uint32_t M = match(w, E, F);
                for (; 32 * t <= dhi; ++t) {
                    ++w;
#pragma unroll
                    for (int k = 0; k < 4; ++k) E[k] = F[k];
                    letter_words(planes(w + 1), c0, c1, F);
                    const uint32_t N = match(w, E, F);
                    f(t, __funnelshift_r(M, N, s));
                    M = N;
                }
            };
            if (2 * W + 1 <= kShortWindow) {
                // A short window has fewer matches than bins: each is taken by
                // itself.  Its bin is floor(64 d / D), from a multiply by 1 / D:
                // 64 d + 0.5 keeps at least 0.5 / D = 2^-9 from the next whole number,
                // the rounding is below 2^-17.
                const uint32_t D = 2u * (uint32_t)W + 1u;
                const float inv = 1.f / (float)D;
                words([&](int32_t at, uint32_t x) {
                    for (; x; x &= x - 1) {
                        const uint32_t d = 32u * (uint32_t)at + (uint32_t)__ffs(x) - 1u;
                        if (d < D) atomicAdd(&hist[(uint32_t)(((float)(d * kBins) + 0.5f) * inv)], 1u);
                    }
                });
            } else {
                const int64_t D = 2 * (int64_t)W + 1;
                uint32_t bin = (uint32_t)((int64_t)t * 32 * kBins / D);
                const auto bin_end = [&](uint32_t b) { return (int32_t)(((int64_t)(b + 1) * D + kBins - 1) / kBins); };
                int32_t end = bin_end(bin);  // the first d past the bin
                uint32_t acc = 0, h0 = 0, h1 = 0;
                const auto flush = [&] {
                    const uint32_t sum = __reduce_add_sync(~0u, acc);
                    if (lane == (bin & 31u)) (bin < 32u ? h0 : h1) = sum;
                };
                words([&](int32_t at, uint32_t x) {
                    while (bin < (uint32_t)kBins && end <= 32 * at + 32) {
                        const uint32_t in = ~0u >> (32 * at + 32 - end);  // end > 32 t
                        acc += __popc(x & in);
                        x &= ~in;
                        flush();
                        acc = 0;
                        end = bin_end(++bin);
                    }
                    acc += __popc(x);
                });
                if (bin < (uint32_t)kBins) flush();
                if (h0) atomicAdd(&hist[lane], h0);
                if (h1) atomicAdd(&hist[lane + 32], h1);
            }
        }
        __syncthreads();
        if (threadIdx.x < kBins) {
            const float norm = K ? log1pf((float)K) : 1.f;
            feat[(size_t)p * kF + threadIdx.x] = log1pf((float)hist[threadIdx.x]) / norm;
        }
        if (threadIdx.x == kBins) feat[(size_t)p * kF + kBins] = L ? (float)delta / (float)L : 0.f;
        __syncthreads();
    }
}

// ---------------------------------------------------------------- network
__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// The network on tiles of kTileB samples, 128 threads: thread u holds unit u of
// the layer at work for every sample of the tile.  The BF16 weights stay in
// shared memory, [input][unit], for all the tiles a CTA takes; the tile's
// inputs and activations are [input][sample], so a step of a layer is one
// weight, two 16-byte broadcasts and eight multiply-adds.  A layer's sum runs
// over its inputs in order, as one thread per (sample, unit) would add them.
//
// GRAD: also dy = (y - t) / B and the layers' errors dh2, dh1 (masked by
// ReLU'), and everything the weight gradients need goes to global memory.
//
// One thread per (sample, unit) read both operands of each multiply-add from
// global memory: nine launches of about 20 us for the gradients of 512 samples,
// 0.66 ms for the outputs of 10,000.
constexpr int kTileB = 8;
constexpr int kWPad = kH + 4;  // a weight row in shared memory

struct NetArgs {
    const float *x;             // n x 65
    uint32_t n;
    const __nv_bfloat16 *wb;
    const float *master;        // biases
    float *y;
    const float *t;             // GRAD: targets, and out: per sample
    float *h1, *h2, *dh1, *dh2, *dy;
};

struct NetShared {
    __nv_bfloat16 w1[kF][kWPad], w2[kH][kWPad], w3[kH];
    alignas(16) float x[kF][kTileB];
    alignas(16) float h1[kH][kTileB];
    alignas(16) float h2[kH][kTileB];
    float dy[kTileB];
};

// acc[s] += sum over k in order of w[k][u] * in[k][s]
template <int K>
__device__ __forceinline__ void net_layer(const __nv_bfloat16 (*w)[kWPad], const float (*in)[kTileB], uint32_t u,
                                          float (&acc)[kTileB]) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float wk = __bfloat162float(w[k][u]);
        const float4 a = *reinterpret_cast<const float4 *>(&in[k][0]), b = *reinterpret_cast<const float4 *>(&in[k][4]);
        acc[0] = fmaf(wk, a.x, acc[0]);
        acc[1] = fmaf(wk, a.y, acc[1]);
        acc[2] = fmaf(wk, a.z, acc[2]);
        acc[3] = fmaf(wk, a.w, acc[3]);
        acc[4] = fmaf(wk, b.x, acc[4]);
        acc[5] = fmaf(wk, b.y, acc[5]);
        acc[6] = fmaf(wk, b.z, acc[6]);
        acc[7] = fmaf(wk, b.w, acc[7]);
    }
}

template <bool GRAD>
__global__ void __launch_bounds__(kH) k_net(NetArgs p) {
    extern __shared__ __align__(16) uint8_t net_smem[];
    NetShared &sm = *reinterpret_cast<NetShared *>(net_smem);
    const uint32_t u = threadIdx.x;
    for (uint32_t q = u; q < (uint32_t)kNW1; q += kH) sm.w1[q % kF][q / kF] = p.wb[kOffW1 + q];
    for (uint32_t q = u; q < (uint32_t)kNW2; q += kH) sm.w2[q % kH][q / kH] = p.wb[kOffW2 + q];
    sm.w3[u] = p.wb[kOffW3 + u];
    const float b1 = p.master[kOffB1 + u], b2 = p.master[kOffB2 + u], b3 = p.master[kOffB3];
    const uint32_t tiles = (p.n + kTileB - 1) / kTileB;
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const uint32_t s0 = tile * kTileB, ns = min((uint32_t)kTileB, p.n - s0);
        __syncthreads();  // the weights, and the last tile's activations read
        for (uint32_t q = u; q < (uint32_t)(kF * kTileB); q += kH) {
            const uint32_t s = q / kF, k = q % kF;
            sm.x[k][s] = s < ns ? bf(p.x[(size_t)(s0 + s) * kF + k]) : 0.f;
        }
        __syncthreads();
        float acc[kTileB] = {};
        net_layer<kF>(sm.w1, sm.x, u, acc);
#pragma unroll
        for (int s = 0; s < kTileB; ++s) {
            const float h = bf(fmaxf(acc[s] + b1, 0.f));
            sm.h1[u][s] = h;
            if (GRAD && (uint32_t)s < ns) p.h1[(size_t)(s0 + s) * kH + u] = h;
            acc[s] = 0.f;
        }
        __syncthreads();
        net_layer<kH>(sm.w2, sm.h1, u, acc);
        float h2[kTileB];
#pragma unroll
        for (int s = 0; s < kTileB; ++s) {
            h2[s] = bf(fmaxf(acc[s] + b2, 0.f));
            sm.h2[u][s] = h2[s];
            if (GRAD && (uint32_t)s < ns) p.h2[(size_t)(s0 + s) * kH + u] = h2[s];
        }
        __syncthreads();
        if (u < ns) {
            float y = 0.f;
            for (int k = 0; k < kH; ++k) y = fmaf(__bfloat162float(sm.w3[k]), sm.h2[k][u], y);
            y += b3;
            p.y[s0 + u] = y;
            if constexpr (GRAD) {
                const float d = (y - p.t[s0 + u]) / (float)p.n;
                sm.dy[u] = d;
                p.dy[s0 + u] = d;
            }
        } else if (GRAD && u < (uint32_t)kTileB) {
            sm.dy[u] = 0.f;
        }
        if constexpr (GRAD) {
            __syncthreads();
            // dh2 = W3 dy where h2 > 0 (over h2 in shared memory: this thread's row)
            const float w3 = __bfloat162float(sm.w3[u]);
#pragma unroll
            for (int s = 0; s < kTileB; ++s) {
                const float d = h2[s] > 0.f ? sm.dy[s] * w3 : 0.f;
                sm.h2[u][s] = d;
                if ((uint32_t)s < ns) p.dh2[(size_t)(s0 + s) * kH + u] = d;
            }
            __syncthreads();
            // dh1 = W2^T dh2 where h1 > 0: this thread's input k = u
            float d1[kTileB] = {};
#pragma unroll 4
            for (int o = 0; o < kH; ++o) {
                const float w = __bfloat162float(sm.w2[u][o]);
                const float4 a = *reinterpret_cast<const float4 *>(&sm.h2[o][0]);
                const float4 b = *reinterpret_cast<const float4 *>(&sm.h2[o][4]);
                d1[0] = fmaf(a.x, w, d1[0]);
                d1[1] = fmaf(a.y, w, d1[1]);
                d1[2] = fmaf(a.z, w, d1[2]);
                d1[3] = fmaf(a.w, w, d1[3]);
                d1[4] = fmaf(b.x, w, d1[4]);
                d1[5] = fmaf(b.y, w, d1[5]);
                d1[6] = fmaf(b.z, w, d1[6]);
                d1[7] = fmaf(b.w, w, d1[7]);
            }
#pragma unroll
            for (int s = 0; s < kTileB; ++s)
                if ((uint32_t)s < ns) p.dh1[(size_t)(s0 + s) * kH + u] = sm.h1[u][s] > 0.f ? d1[s] : 0.f;
        }
    }
}

// Weight gradients of a share of the samples: dW[u][k] = sum_b d[b][u] in[b][k],
// dbias[u] = sum_b d[b][u], and the loss.  blockIdx.x: 16 units of layer 2 or
// layer 1, or layer 3; blockIdx.y: the share, whose sums go to its own row of
// `part`.
constexpr int kUnits = 16;
__global__ void __launch_bounds__(kH) k_net_weights(NetArgs p, uint32_t per, float *part) {
    __shared__ float d[32][kUnits];
    const uint32_t k = threadIdx.x, tiles = kH / kUnits;
    const uint32_t b0 = blockIdx.y * per, b1 = min(p.n, b0 + per);
    float *out = part + (size_t)blockIdx.y * (kNParams + 1);
    if (blockIdx.x == 2 * tiles) {  // layer 3 and the loss
        float acc = 0.f, db = 0.f, loss = 0.f;
        for (uint32_t b = b0; b < b1; ++b) acc = fmaf(p.dy[b], p.h2[(size_t)b * kH + k], acc);
        out[kOffW3 + k] = acc;
        if (k < 32) {
            for (uint32_t b = b0 + k; b < b1; b += 32) {
                const float e = p.y[b] - p.t[b];
                db += p.dy[b];
                loss += 0.5f * e * e / (float)p.n;
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                db += __shfl_xor_sync(0xffffffffu, db, o);
                loss += __shfl_xor_sync(0xffffffffu, loss, o);
            }
            if (k == 0) {
                out[kOffB3] = db;
                out[kNParams] = loss;
            }
        }
        return;
    }
    const bool two = blockIdx.x < tiles;
    const uint32_t u0 = (blockIdx.x % tiles) * kUnits, nin = two ? kH : kF;
    const float *err = two ? p.dh2 : p.dh1;
    float acc[kUnits] = {}, bias = 0.f;
    for (uint32_t c = b0; c < b1; c += 32) {
        const uint32_t nb = min(32u, b1 - c);
        __syncthreads();
        for (uint32_t q = k; q < 32u * kUnits; q += kH)
            d[q / kUnits][q % kUnits] = q / kUnits < nb ? err[(size_t)(c + q / kUnits) * kH + u0 + q % kUnits] : 0.f;
        __syncthreads();
        if (k < (uint32_t)kUnits)
            for (uint32_t b = 0; b < nb; ++b) bias += d[b][k];
        if (k < nin) {
#pragma unroll 4
            for (uint32_t b = 0; b < nb; ++b) {
                const float in = two ? p.h1[(size_t)(c + b) * kH + k] : bf(p.x[(size_t)(c + b) * kF + k]);
#pragma unroll
                for (int q = 0; q < kUnits; ++q) acc[q] = fmaf(d[b][q], in, acc[q]);
            }
        }
    }
    if (k < nin)
#pragma unroll
        for (int q = 0; q < kUnits; ++q) out[(two ? kOffW2 : kOffW1) + (u0 + q) * nin + k] = acc[q];
    if (k < (uint32_t)kUnits) out[(two ? kOffB2 : kOffB1) + u0 + k] = bias;
}

// The shares' sums.
__global__ void k_net_sum(const float *part, uint32_t shares, float *grad, float *loss) {
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q > (uint32_t)kNParams) return;
    float acc = 0.f;
    for (uint32_t s = 0; s < shares; ++s) acc += part[(size_t)s * (kNParams + 1) + q];
    if (q < (uint32_t)kNParams) grad[q] = acc;
    else *loss = acc;
}

__global__ void k_adam(float *p, const float *g, float *m, float *v, int n, float lr, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = 0.9f * m[i] + 0.1f * gi;
    const float vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

__global__ void k_refresh_bf16(const float *p, __nv_bfloat16 *wb, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) wb[i] = __float2bfloat16_rn(p[i]);
}

// He-style initialisation from a counter-based SplitMix64 stream: value k
// is mix64(seed + (k+1) * 0x9E3779B97F4A7C15), mapped to a uniform in
// [-1, 1) and scaled by sqrt(6 / fan_in); biases start at 0 except b3.
__device__ __forceinline__ uint64_t splitmix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_init(float *p, uint64_t seed, float b3) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kNParams) return;
    float fan = 0.f;
    if (i < kOffB1) fan = kF;
    else if (i >= kOffW2 && i < kOffB2) fan = kH;
    else if (i >= kOffW3 && i < kOffB3) fan = kH;
    if (fan == 0.f) {
        p[i] = i == kOffB3 ? b3 : 0.f;
        return;
    }
    const uint64_t r = splitmix(seed + (uint64_t)(i + 1) * 0x9E3779B97F4A7C15ull);
    const float u = (float)((double)(r >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;
    p[i] = u * sqrtf(6.f / fan);
}

// ------------------------------------------------------------------- host
static unsigned blocks_for(uint64_t n, unsigned t = 256) { return (unsigned)((n + t - 1) / t); }

static int model_of(nw_ctx *ctx, BandModel **out, bool create) {
    if (!ctx->band_model) {
        if (!create) return fail(ctx, NW_ERR_ARG, "no band model: call nw_band_model_init or nw_band_model_set");
        BandModel *bm = new BandModel();
        cudaError_t e = cudaMalloc(&bm->master, kNParams * 4);
        if (e == cudaSuccess) e = cudaMalloc(&bm->wb, kNParams * 2);
        if (e == cudaSuccess) e = cudaMalloc(&bm->adam_m, kNParams * 4);
        if (e == cudaSuccess) e = cudaMalloc(&bm->adam_v, kNParams * 4);
        if (e == cudaSuccess) e = cudaMalloc(&bm->grad, (kNParams + 1) * 4);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(ctx, NW_ERR_OOM, "band model allocation failed");
        }
        cudaMemsetAsync(bm->adam_m, 0, kNParams * 4, ctx->stream);
        cudaMemsetAsync(bm->adam_v, 0, kNParams * 4, ctx->stream);
        ctx->band_model = bm;
    }
    *out = (BandModel *)ctx->band_model;
    return NW_OK;
}

void free_band_model(nw_ctx *ctx) {
    BandModel *bm = (BandModel *)ctx->band_model;
    if (!bm) return;
    cudaFree(bm->master);
    cudaFree(bm->wb);
    cudaFree(bm->adam_m);
    cudaFree(bm->adam_v);
    cudaFree(bm->grad);
    delete bm;
    ctx->band_model = nullptr;
}

static void refresh(nw_ctx *ctx, BandModel *bm) {
    k_refresh_bf16<<<blocks_for(kNParams), 256, 0, ctx->stream>>>(bm->master, bm->wb, kNParams);
}

static constexpr int kNetSmem = (int)sizeof(NetShared);

static int launch_net(nw_ctx *ctx, const NetArgs &a, bool grad) {
    const void *kern = grad ? (const void *)k_net<true> : (const void *)k_net<false>;
    // one value for every caller: the attribute belongs to the process
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kNetSmem);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "network shared memory");
    const uint32_t tiles = (a.n + kTileB - 1) / kTileB;
    // three CTAs fit an SM's shared memory; more tiles reuse the weights a CTA holds
    const uint32_t blocks = std::min<uint32_t>(tiles, 3u * (uint32_t)ctx->sm_count);
    if (grad) k_net<true><<<blocks, kH, kNetSmem, ctx->stream>>>(a);
    else k_net<false><<<blocks, kH, kNetSmem, ctx->stream>>>(a);
    e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "network launch");
}

// Outputs for n feature rows.
static int forward(nw_ctx *ctx, BandModel *bm, const float *x, uint32_t n, float *y) {
    NetArgs a{};
    a.x = x;
    a.n = n;
    a.wb = bm->wb;
    a.master = bm->master;
    a.y = y;
    LaunchTimer t(ctx, "mlp_forward", 1);
    return launch_net(ctx, a, false);
}

// Gradients into grad (kNParams) and the loss.
static int gradients(nw_ctx *ctx, BandModel *bm, const float *x, const float *t, uint32_t nb, float *grad, float *loss) {
    // Shares of at least 32 samples, as many as the scratch has room for (100 KB
    // each beside the activations); one share's sums fit the model's own
    // gradients.
    const size_t acts = (size_t)nb * (4 * kH + 2) * 4 + 64, one = (size_t)(kNParams + 1) * 4;
    const uint64_t room = scratch_headroom(ctx, "mlp_acts");
    uint32_t per = std::max<uint32_t>(32, (nb + 31) / 32), shares = (nb + per - 1) / per;
    if (acts + shares * one > room) {
        shares = (uint32_t)std::max<uint64_t>(1, (room - std::min<uint64_t>(room, acts)) / one);
        per = (nb + shares - 1) / shares;
        shares = (nb + per - 1) / per;
    }
    const bool in_model = acts + shares * one > room;
    void *v = nullptr;
    int rc = scratch(ctx, "mlp_acts", acts + (in_model ? 0 : shares * one), &v);
    if (rc) return rc;
    NetArgs a{};
    a.x = x;
    a.n = nb;
    a.wb = bm->wb;
    a.master = bm->master;
    a.t = t;
    a.h1 = (float *)v;
    a.h2 = a.h1 + (size_t)nb * kH;
    a.dh1 = a.h2 + (size_t)nb * kH;
    a.dh2 = a.dh1 + (size_t)nb * kH;
    a.dy = a.dh2 + (size_t)nb * kH;
    a.y = a.dy + nb;
    float *part = in_model ? bm->grad : a.y + nb;
    {
        LaunchTimer lt(ctx, "mlp_forward", 1);
        if ((rc = launch_net(ctx, a, true))) return rc;
    }
    LaunchTimer lt(ctx, "mlp_backward", 2);
    k_net_weights<<<dim3(2 * (kH / kUnits) + 1, shares), kH, 0, ctx->stream>>>(a, per, part);
    k_net_sum<<<blocks_for(kNParams + 1), 256, 0, ctx->stream>>>(part, shares, grad, loss);
    return NW_OK;
}

}  // namespace nw

using namespace nw;

// The feature kernel keeps B's bit planes in dynamic shared memory, 8 bytes
// per 32 bases.  Its limit above the default 48 KiB is a per-function
// attribute of the process, which concurrent callers (the server's workers)
// share: it is always set to the one value that covers every accepted B, never
// to a call's own need, so a launch never meets a smaller limit set by another
// thread.
constexpr uint32_t kFeatMaxB = 200000;
constexpr size_t feature_bytes(uint32_t n) { return (size_t)(n + 31) / 32 * sizeof(uint2); }

static int launch_features(nw_ctx *ctx, const uint8_t *pool, const uint64_t *a_off, const uint32_t *a_len,
                           const uint64_t *b_off, const uint32_t *b_len, uint32_t npairs, uint32_t maxn, float *feat) {
    // (the default limit counts the kernel's static words too)
    if (feature_bytes(maxn) + kBins * sizeof(uint32_t) > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_features<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)feature_bytes(kFeatMaxB));
        if (e != cudaSuccess) return cuda_fail(ctx, e, "feature kernel shared memory");
    }
    {
        LaunchTimer t(ctx, "features");
        // Short pairs are a chain of loads and barriers, so an SM holds eight CTAs (32
        // registers a thread, a few spilled); longer ones take the 48 registers.
        // 100,000 pairs of 50 to 150 bases .50 ms against .71; 10,000 of 2 kb .38 against
        // .37.
        const auto kern = maxn < 1024 ? k_features<8> : k_features<1>;
        kern<<<std::min<uint32_t>(npairs, (uint32_t)ctx->sm_count * 8), kAnchors, feature_bytes(maxn),
                     ctx->stream>>>(pool, a_off, a_len, b_off, b_len, npairs, feat);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "features launch");
}

// Features -> network -> half-widths (with a safety factor), on the host.
uint32_t band_start_width(float y, uint32_t m, uint32_t n, double margin, double probe_cap, bool skip);

// `overlap` runs on the host once the feature and network kernels are
// queued, before the copy of their output (a copy into pageable memory
// returns only when it is done); not at all when the call keeps the fixed
// start.
int learned_band_widths(nw_ctx *ctx, const uint8_t *pool, const uint64_t *a_off, const uint32_t *a_len,
                        const uint64_t *b_off, const uint32_t *b_len, uint32_t npairs, std::vector<uint32_t> &w,
                        const std::function<int()> &overlap) {
    w.assign(npairs, 64u);
    BandModel *bm = nullptr;
    if (!ctx->band_model) return NW_OK;  // no model: fixed starting width 64
    // The first round's width is 0.75x the predicted one: a round that fails
    // its certificate is followed by one at the smallest width the failed
    // score proves sufficient, so under-predicting costs one narrow pass
    // while over-predicting widens every band.  Effective GCUPS on GB300 (20,000
    // pairs of 2-20 kb): 0.25 -> 58,300, 0.5 -> 56,700, 0.75 -> 55,000, 1 -> 52,500,
    // against 60,600 from the fixed start 64: the first round costs more than the
    // second it saves.  0.75 is the smallest margin at which the network certifies
    // more pairs in the first round than the fixed start on held-out pairs while
    // sweeping fewer banded cells there.  NW_BAND_MARGIN and NW_BAND_PROBE_CAP for
    // sweeps.
    double margin = 0.75;
    if (const char *e = getenv("NW_BAND_MARGIN")) margin = std::max(0.25, atof(e));
    int rc = model_of(ctx, &bm, false);
    if (rc) return rc;
    void *v = nullptr;
    if ((rc = scratch(ctx, "lb_meta", (size_t)npairs * 24 + 64, &v))) return rc;
    uint64_t *dao = (uint64_t *)v, *dbo = dao + npairs;
    uint32_t *dal = (uint32_t *)(dbo + npairs), *dbl = dal + npairs;
    cudaMemcpyAsync(dao, a_off, (size_t)npairs * 8, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(dbo, b_off, (size_t)npairs * 8, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(dal, a_len, (size_t)npairs * 4, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(dbl, b_len, (size_t)npairs * 4, cudaMemcpyHostToDevice, ctx->stream);
    void *f = nullptr;
    if ((rc = scratch(ctx, "lb_feat", (size_t)npairs * kF * 4 + 64, &f))) return rc;
    uint32_t maxn = 4;
    for (uint32_t k = 0; k < npairs; ++k) maxn = std::max(maxn, b_len[k]);
    if (maxn > kFeatMaxB) return NW_OK;  // features need B <= 200,000 bases: keep the fixed start
    if ((rc = launch_features(ctx, pool, dao, dal, dbo, dbl, npairs, maxn, (float *)f))) return rc;
    void *yv = nullptr;
    if ((rc = scratch(ctx, "lb_y", (size_t)npairs * 4 + 64, &yv))) return rc;
    if ((rc = forward(ctx, bm, (const float *)f, npairs, (float *)yv))) return rc;
    if (overlap && (rc = overlap())) return rc;
    std::vector<float> y(npairs);
    cudaMemcpyAsync(y.data(), yv, (size_t)npairs * 4, cudaMemcpyDeviceToHost, ctx->stream);
    if ((rc = nw_ctx_sync(ctx))) return rc;
    // Probe cap (NW_BAND_PROBE_CAP, 0 = none) and the straight-to-full rule
    // (NW_BAND_SKIP: a pair whose predicted band would cover most of the
    // grid starts at that width, which sends it to the full kernel).
    double probe_cap = 0.0;
    if (const char *e = getenv("NW_BAND_PROBE_CAP")) probe_cap = atof(e);
    const bool skip = getenv("NW_BAND_SKIP") != nullptr;
    for (uint32_t k = 0; k < npairs; ++k) w[k] = band_start_width(y[k], a_len[k], b_len[k], margin, probe_cap, skip);
    return NW_OK;
}

// First half-width of a pair from the network's output y = log w:
// ceil(margin * e^y), clamped to [8, max(m, n)].  (Sweep knobs: a probe cap
// on the width, and the straight-to-full rule for a predicted band that would
// cover most of the grid.)
uint32_t band_start_width(float y, uint32_t m, uint32_t n, double margin, double probe_cap, bool skip) {
    const double full_pred = std::exp((double)y);
    double pred = full_pred * margin;
    const double cap = (double)std::max(m, n);
    const double delta = std::fabs((double)n - (double)m);
    if (skip && (512.0 + 2.0 * full_pred + delta) * 20.0 >= (double)n * 17.0) pred = cap;
    else if (probe_cap > 0 && pred > probe_cap) pred = probe_cap;
    return (uint32_t)std::min(cap, std::max(8.0, std::ceil(pred)));
}

extern "C" {

int nw_band_features(nw_ctx *ctx, const uint8_t *pool2b, const uint64_t *a_off, const uint32_t *a_len,
                     const uint64_t *b_off, const uint32_t *b_len, uint32_t npairs, float *feat) {
    if (!ctx) return NW_ERR_ARG;
    if (npairs == 0) return NW_OK;
    if (!pool2b || !a_off || !a_len || !b_off || !b_len || !feat) return fail(ctx, NW_ERR_ARG, "null argument");
    cudaSetDevice(ctx->device);
    void *v = nullptr;
    int rc = scratch(ctx, "feat_meta", (size_t)npairs * 24 + 64, &v);
    if (rc) return rc;
    uint64_t *dao = (uint64_t *)v, *dbo = dao + npairs;
    uint32_t *dal = (uint32_t *)(dbo + npairs), *dbl = dal + npairs;
    cudaMemcpyAsync(dao, a_off, (size_t)npairs * 8, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(dbo, b_off, (size_t)npairs * 8, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(dal, a_len, (size_t)npairs * 4, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(dbl, b_len, (size_t)npairs * 4, cudaMemcpyHostToDevice, ctx->stream);
    uint32_t maxn = 4;
    for (uint32_t k = 0; k < npairs; ++k) maxn = std::max(maxn, b_len[k]);
    if (maxn > kFeatMaxB) return fail(ctx, NW_ERR_ARG, "features need B <= 200,000 bases");
    if ((rc = launch_features(ctx, pool2b, dao, dal, dbo, dbl, npairs, maxn, feat))) return rc;
    // the metadata copies read host arrays the caller may free on return
    const cudaError_t e = cudaStreamSynchronize(ctx->stream);
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "features sync");
}

int nw_band_model_init(nw_ctx *ctx, uint64_t seed) {
    if (!ctx) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    BandModel *bm = nullptr;
    int rc = model_of(ctx, &bm, true);
    if (rc) return rc;
    k_init<<<blocks_for(kNParams), 256, 0, ctx->stream>>>(bm->master, seed, std::log(64.f));
    cudaMemsetAsync(bm->adam_m, 0, kNParams * 4, ctx->stream);
    cudaMemsetAsync(bm->adam_v, 0, kNParams * 4, ctx->stream);
    bm->step = 0;
    refresh(ctx, bm);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "model init");
}

uint32_t nw_band_start_width(float y, uint64_t m, uint64_t n) {
    if (m >= (1ull << 31) || n >= (1ull << 31)) return 0;
    return band_start_width(y, (uint32_t)m, (uint32_t)n, 0.75, 0.0, false);
}

uint64_t nw_band_model_size(void) { return kNParams; }

int nw_band_model_set(nw_ctx *ctx, const float *params, uint64_t count) {
    if (!ctx || !params || count != (uint64_t)kNParams) return ctx ? fail(ctx, NW_ERR_ARG, "need %d params", kNParams) : NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    BandModel *bm = nullptr;
    int rc = model_of(ctx, &bm, true);
    if (rc) return rc;
    cudaMemcpyAsync(bm->master, params, kNParams * 4, cudaMemcpyHostToDevice, ctx->stream);
    refresh(ctx, bm);
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "model set");
}

// File format of a saved model: the 8 bytes "NWBAND01", the parameter
// count as a little-endian uint64, then the FP32 master parameters in the
// layout nw_band_model_get returns (little-endian IEEE-754).
int nw_band_model_save(nw_ctx *ctx, const char *path) {
    if (!ctx || !path) return NW_ERR_ARG;
    std::vector<float> p(kNParams);
    int rc = nw_band_model_get(ctx, p.data(), p.size());
    if (rc) return rc;
    FILE *f = fopen(path, "wb");
    if (!f) return fail(ctx, NW_ERR_ARG, "cannot open '%s' for writing", path);
    const uint64_t count = kNParams;
    const bool ok = fwrite("NWBAND01", 1, 8, f) == 8 && fwrite(&count, 8, 1, f) == 1 &&
                    fwrite(p.data(), 4, p.size(), f) == p.size();
    const bool closed = fclose(f) == 0;
    return ok && closed ? NW_OK : fail(ctx, NW_ERR_ARG, "short write to '%s'", path);
}

int nw_band_model_load(nw_ctx *ctx, const char *path) {
    if (!ctx || !path) return NW_ERR_ARG;
    FILE *f = fopen(path, "rb");
    if (!f) return fail(ctx, NW_ERR_ARG, "cannot open '%s'", path);
    char magic[8] = {0};
    uint64_t count = 0;
    std::vector<float> p(kNParams);
    const bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, "NWBAND01", 8) == 0 && fread(&count, 8, 1, f) == 1 &&
                    count == (uint64_t)kNParams && fread(p.data(), 4, p.size(), f) == p.size() && fgetc(f) == EOF;
    fclose(f);
    if (!ok) return fail(ctx, NW_ERR_ARG, "'%s' is not a saved band model of %d parameters", path, kNParams);
    return nw_band_model_set(ctx, p.data(), p.size());
}

int nw_band_model_clear(nw_ctx *ctx) {
    if (!ctx) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    cudaError_t e = cudaStreamSynchronize(ctx->stream);  // no kernel still reads the parameters
    free_band_model(ctx);
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "model clear");
}

int nw_band_model_get(nw_ctx *ctx, float *params, uint64_t count) {
    if (!ctx || !params || count != (uint64_t)kNParams) return ctx ? fail(ctx, NW_ERR_ARG, "need %d params", kNParams) : NW_ERR_ARG;
    BandModel *bm = nullptr;
    int rc = model_of(ctx, &bm, false);
    if (rc) return rc;
    cudaMemcpyAsync(params, bm->master, kNParams * 4, cudaMemcpyDeviceToHost, ctx->stream);
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "model get");
}

int nw_band_model_forward(nw_ctx *ctx, const float *feat, uint32_t n, float *out) {
    if (!ctx || (n && (!feat || !out))) return NW_ERR_ARG;
    if (!n) return NW_OK;
    cudaSetDevice(ctx->device);
    BandModel *bm = nullptr;
    int rc = model_of(ctx, &bm, false);
    if (rc) return rc;
    // outputs that lie in the inputs (the kernel writes a tile's before others are read)
    const uintptr_t f0 = (uintptr_t)feat, f1 = f0 + (size_t)n * kF * 4, o0 = (uintptr_t)out, o1 = o0 + (size_t)n * 4;
    if (o0 >= f1 || f0 >= o1) return forward(ctx, bm, feat, n, out);
    void *y = nullptr;
    if ((rc = scratch(ctx, "mlp_acts", (size_t)n * 4, &y)) || (rc = forward(ctx, bm, feat, n, (float *)y))) return rc;
    const cudaError_t e = cudaMemcpyAsync(out, y, (size_t)n * 4, cudaMemcpyDeviceToDevice, ctx->stream);
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "model forward");
}

int nw_band_model_grad(nw_ctx *ctx, const float *feat, const float *target, uint32_t n, float *grad, float *loss) {
    if (!ctx || !feat || !target || !grad || !loss || !n) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    BandModel *bm = nullptr;
    int rc = model_of(ctx, &bm, false);
    if (rc) return rc;
    if ((rc = gradients(ctx, bm, feat, target, n, grad, loss))) return rc;
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "model grad");
}

int nw_band_model_train_step(nw_ctx *ctx, const float *feat, const float *target, uint32_t n, float lr, float *loss) {
    if (!ctx || !feat || !target || !loss || !n) return NW_ERR_ARG;
    cudaSetDevice(ctx->device);
    BandModel *bm = nullptr;
    int rc = model_of(ctx, &bm, false);
    if (rc) return rc;
    if ((rc = gradients(ctx, bm, feat, target, n, bm->grad, loss))) return rc;
    bm->step += 1;
    const float c1 = 1.f - std::pow(0.9f, (float)bm->step), c2 = 1.f - std::pow(0.999f, (float)bm->step);
    {
        LaunchTimer t(ctx, "adam");
        k_adam<<<blocks_for(kNParams), 256, 0, ctx->stream>>>(bm->master, bm->grad, bm->adam_m, bm->adam_v, kNParams,
                                                               lr, c1, c2);
    }
    refresh(ctx, bm);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NW_OK : cuda_fail(ctx, e, "train step");
}

}  // extern "C"
