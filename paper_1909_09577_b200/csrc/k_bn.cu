// Lengths, masked batch-norm statistics / apply / backward, and small elementwise kernels.
// All of these stream [B,C,T] tensors once; one CTA handles one (sample, channel) row so that the
// per-channel coefficients are loaded once and reductions stay inside the CTA (warp shuffles +
// one shared-memory step).  Cross-CTA reductions go through per-row partials that a finalize
// kernel sums in a fixed order, so results are bit-repeatable.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace sc {
namespace {

constexpr int kRowThreads = 256;          // 8 warps per CTA, one (sample, channel) row per warp
constexpr int kRowsPerCta = kRowThreads / 32;
#define SC_ROW_SETUP(nrows)                                                  \
    const int row = blockIdx.x * kRowsPerCta + (threadIdx.x >> 5);          \
    if (row >= (nrows)) return;                                              \
    const int lane = threadIdx.x & 31;

template <typename T>
__device__ __forceinline__ void load_chunk(const T* row, int t0, int Tp, bool vec, float (&f)[8]) {
    if (vec && t0 + 8 <= Tp) { ld8<T>(row + t0, f); return; }
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = (t0 + i < Tp) ? ldf(row + t0 + i) : 0.f;
}
template <typename T>
__device__ __forceinline__ void store_chunk(T* row, int t0, int Tp, bool vec, const float (&f)[8]) {
    if (vec && t0 + 8 <= Tp) { st8<T>(row + t0, f); return; }
#pragma unroll
    for (int i = 0; i < 8; ++i) if (t0 + i < Tp) stf(row + t0 + i, f[i]);
}

// Sum of `v` over the warp that owns the row; result valid in every lane.
template <int N>
__device__ __forceinline__ void block_sum(float (&v)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = warp_sum(v[i]);
}

__device__ __forceinline__ float block_max(float v) { return warp_max(v); }

// Block 0: lengths.  The block offsets are an exclusive scan over the samples: each thread sums a contiguous run of
// samples, the runs are scanned through shared memory.  (A scan by one thread is a chain of dependent loads: 10 us at 32
// samples.)  The other blocks convert 2048 elements each, one 16-byte vector per thread; as a launch of its own with scalar
// accesses the conversion of an encoder's weights cost 12 us in front of every training step.
constexpr int kLenThreads = 256, kConvertChunk = 2048;
__global__ void __launch_bounds__(kLenThreads) prologue_kernel(const __grid_constant__ Prologue p, int* status) {
    pdl_sync();
    const int tid = threadIdx.x;
    if (blockIdx.x > 0) {
        const ConvertList& l = p.conv;
        const int blk = blockIdx.x - 1;
        int k = 0;
        while (k + 1 < l.count && blk >= l.first[k + 1]) ++k;
        const int i = (blk - l.first[k]) * kConvertChunk + 8 * tid, n = l.n[k];
        const __nv_bfloat16* src = (const __nv_bfloat16*)l.src[k];
        __half* dst = (__half*)l.dst[k];
        if (i + 8 <= n && ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
            float f[8];
            ld8<__nv_bfloat16>(src + i, f);
            st8<__half>(dst + i, f);
        } else {
            for (int e = i; e < min(i + 8, n); ++e) dst[e] = __float2half_rn(__bfloat162float(src[e]));
        }
        return;
    }
    for (int i = tid; i < p.nzero; i += kLenThreads) p.zero[i] = 0.f;
    if (!p.len_in) return;
    __shared__ int s_frames[kLenThreads / 32], s_blocks[kLenThreads / 32];
    const int lane = tid & 31, w = tid >> 5;
    const int n = p.B * p.phases, per = (n + kLenThreads - 1) / kLenThreads, i0 = min(n, tid * per), i1 = min(n, i0 + per);
    int frames = 0, blocks = 0;
    for (int i = i0; i < i1; ++i) {
        const int b = i / p.phases, ph = i - b * p.phases;
        int l = p.len_in[b];
        if (l < 1 || l > p.T_in) { raise_status(status, kErrLengths); l = min(max(l, 0), p.T_in); }
        const int lo = p.phases > 1 ? (l - ph + p.phases - 1) / p.phases : (l + p.stride - 1) / p.stride;
        if (ph == 0) {
            const int dense = p.phases > 1 ? l : lo;
            if (p.len_dense) p.len_dense[b] = dense;
            if (p.len_user) p.len_user[b] = dense;
        }
        p.len_out[i] = lo;
        frames += lo; blocks += (lo + 63) / 64;
    }
    int incl = blocks;                                   // inclusive scan over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int q = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += q; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) frames += __shfl_xor_sync(0xffffffffu, frames, o);
    if (lane == 31) s_blocks[w] = incl;
    if (lane == 0) s_frames[w] = frames;
    __syncthreads();
    int base = incl - blocks;
    for (int q = 0; q < w; ++q) base += s_blocks[q];
    if (p.blk_off) {
        for (int i = i0; i < i1; ++i) { p.blk_off[i] = base; base += (p.len_out[i] + 63) / 64; }
        if (tid == kLenThreads - 1) p.blk_off[n] = base; // the last thread's runs end the list
    }
    if (tid == 0) {
        int t = 0;
        for (int q = 0; q < kLenThreads / 32; ++q) t += s_frames[q];
        *p.nvalid = t;
    }
}

template <typename T>
__global__ void __launch_bounds__(kRowThreads)
bn_stats_kernel(const T* __restrict__ v, const int* __restrict__ len_out, int nrows, int C, int Tp,
                float2* __restrict__ partials) {
    pdl_sync();
    SC_ROW_SETUP(nrows)
    const int b = row / C;
    const int len = min(len_out[b], Tp);
    const T* p = v + (size_t)row * Tp;
    const bool vec = (Tp % 8 == 0);
    float s[1] = {0.f};
    for (int t0 = lane * 8; t0 < len; t0 += 256) {
        float f[8];
        load_chunk(p, t0, Tp, vec, f);
#pragma unroll
        for (int i = 0; i < 8; ++i) if (t0 + i < len) s[0] += f[i];
    }
    block_sum(s);
    const float mean = len > 0 ? s[0] / (float)len : 0.f;
    float q[1] = {0.f};
    for (int t0 = lane * 8; t0 < len; t0 += 256) {
        float f[8];
        load_chunk(p, t0, Tp, vec, f);
#pragma unroll
        for (int i = 0; i < 8; ++i) if (t0 + i < len) { float d = f[i] - mean; q[0] += d * d; }
    }
    block_sum(q);
    if (lane == 0) partials[row] = make_float2(s[0], q[0]);
}

// Thirty-two channels per CTA, one per lane, so that every load of a warp is one contiguous run of the
// [part][channel] partial array.  Warp w takes parts w, w + 32, ... in increasing order; the thirty-two
// warp results are combined in warp order, so the result is bit-repeatable.  One pass: with a pivot c
// (the mean of the channel's first part, which always holds at least one valid frame)
//   sum = sum_p sum_p,   M2 = sum_p [M2_p + n_p (mean_p - c)^2]  -  N (mean - c)^2,
// and because c lies within the spread of the data the subtraction cancels nothing that matters.
// No term depends on the previous one, so a lane's few loads are all in flight together.
constexpr int kFinWarps = 32;
__global__ void __launch_bounds__(32 * kFinWarps)
bn_finalize_kernel(const float2* __restrict__ partials, int parts_per_b, int tile_w,
                   const int* __restrict__ len_out, const int* __restrict__ nvalid, int B,
                   int C, float eps, float momentum, float* __restrict__ mean_out,
                   float* __restrict__ invstd_out, float* running_mean, float* running_var) {
    pdl_sync();
    __shared__ float2 s_red[kFinWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    const bool act = o < C;
    const int nparts = B * parts_per_b;
    auto count_of = [&](int pi) -> int {
        const int b = pi / parts_per_b, j = pi - b * parts_per_b;
        return max(0, min(len_out[b] - j * tile_w, tile_w));
    };
    float s1 = 0.f, q = 0.f;
    if (act) {
        const float c = partials[o].x / (float)max(1, count_of(0));
        for (int p0 = w; p0 < nparts; p0 += 8 * kFinWarps) {
            float2 v[8]; int cnt[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {        // issue every load before the first use
                const int pi = p0 + i * kFinWarps;
                cnt[i] = pi < nparts ? count_of(pi) : 0;
                v[i] = cnt[i] > 0 ? partials[(size_t)pi * C + o] : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (cnt[i] > 0) {
                    const float n = (float)cnt[i];
                    const float d = v[i].x / n - c;
                    s1 += v[i].x;
                    q += fmaf(n * d, d, v[i].y);
                }
            }
        }
    }
    s_red[w][lane] = make_float2(s1, q);
    __syncthreads();
    if (w != 0 || !act) return;
    // the tail runs in float: a double divide and square root would cost this latency-bound kernel more than the
    // whole merge, and the pivot keeps the subtraction below free of cancellation
    const float N = (float)(*nvalid);
    const float c = partials[o].x / (float)max(1, count_of(0));
    float t = 0.f, m2 = 0.f;
#pragma unroll
    for (int i = 0; i < kFinWarps; ++i) { t += s_red[i][lane].x; m2 += s_red[i][lane].y; }
    const float mean = N > 0.f ? t / N : 0.f;
    const float dm = mean - c;
    float var = N > 0.f ? (m2 - N * dm * dm) / N : 0.f;
    var = fmaxf(var, 0.f);
    mean_out[o] = mean;
    invstd_out[o] = 1.f / sqrtf(var + eps);
    if (running_mean) running_mean[o] = (1.f - momentum) * running_mean[o] + momentum * mean;
    if (running_var) {
        const float unb = N > 1.f ? var * (N / (N - 1.f)) : var;
        running_var[o] = (1.f - momentum) * running_var[o] + momentum * unb;
    }
}

// The same merge for the per-(CTA, channel) partials (count, sum, M2) of the flattened-block contraction.
// CTA c of the contraction contributed to M tile m iff its unit range [c U / G, (c+1) U / G) meets
// [m nblk, (m+1) nblk); the pivot is the mean of the first contributing CTA's partial.
// Unit x belongs to CTA ((x + 1) G - 1) / U, so the contributors are the CTAs between the owners of the tile's first and last
// unit, without those that have no unit at all (only when U < G).  Two divisions; testing every CTA's range took twenty.
struct FlatShare {
    int first, last, G; uint32_t U; bool sparse;
    __device__ __forceinline__ FlatShare(int nblk, int tiles_m, int G_, int m) : G(G_) {
        const long long u = (long long)tiles_m * nblk, lo = (long long)m * nblk, hi = lo + nblk;
        first = 0; last = -1; U = (uint32_t)u; sparse = u < G;
        if (u <= 0) return;
        if (u * (G + 1) < (1ll << 31)) {               // the same quotients in 32-bit arithmetic
            first = (int)((((uint32_t)lo + 1u) * (uint32_t)G - 1u) / U); last = (int)(((uint32_t)hi * (uint32_t)G - 1u) / U);
        } else {
            first = (int)(((lo + 1) * G - 1) / u); last = (int)((hi * G - 1) / u);
        }
    }
    __device__ __forceinline__ bool takes_part(int c) const {
        return c >= first && c <= last && (!sparse || (uint32_t)c * U / (uint32_t)G != ((uint32_t)c + 1u) * U / (uint32_t)G);
    }
};
// sum t and M2 about the pivot -> mean and variance
__device__ __forceinline__ void merged_stats(float N, float t, float m2, float pivot, float& mean, float& var) {
    mean = N > 0.f ? t / N : 0.f;
    const float dm = mean - pivot;
    var = fmaxf(N > 0.f ? (m2 - N * dm * dm) / N : 0.f, 0.f);
}
__device__ __forceinline__ void put_stats(int o, float mean, float invstd, float var, float N, float momentum, float* mean_out, float* invstd_out,
                                          float* running_mean, float* running_var) {
    mean_out[o] = mean;
    invstd_out[o] = invstd;
    if (running_mean) running_mean[o] = (1.f - momentum) * running_mean[o] + momentum * mean;
    if (running_var) running_var[o] = (1.f - momentum) * running_var[o] + momentum * (N > 1.f ? var * (N / (N - 1.f)) : var);
}
constexpr int kFlatParts = 10;        // partials per lane: the contraction has at most 320 CTAs
__global__ void __launch_bounds__(32 * kFinWarps)
bn_finalize_flat_kernel(const float4* __restrict__ partials, int G, int tiles_m, int rows_per_tile,
                        const int* __restrict__ blk_off, const int* __restrict__ nvalid, int B, int C, float eps,
                        float momentum, float* __restrict__ mean_out, float* __restrict__ invstd_out,
                        float* running_mean, float* running_var) {
    __shared__ float2 s_red[kFinWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    const bool act = o < C;
    const FlatShare F(blk_off[B], tiles_m, G, min(o, C - 1) / rows_per_tile);
    // everything above works on the lengths alone and runs ahead of the wait for the contraction; after it the pivot and
    // the partials are one round of independent loads
    uint32_t part = 0;
#pragma unroll
    for (int i = 0; i < kFlatParts; ++i) {
        const int c = w + i * kFinWarps;
        if (act && F.takes_part(c)) part |= 1u << i;
    }
    const float N = (float)(*nvalid);
    pdl_sync();
    float4 pv = make_float4(0.f, 0.f, 0.f, 0.f), v[kFlatParts];
    if (act && F.last >= 0) pv = partials[(size_t)F.first * C + o];
#pragma unroll
    for (int i = 0; i < kFlatParts; ++i)
        v[i] = (part >> i) & 1 ? partials[(size_t)(w + i * kFinWarps) * C + o] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float pivot = pv.x > 0.f ? pv.y / pv.x : 0.f;
    float s1 = 0.f, q = 0.f;
#pragma unroll
    for (int i = 0; i < kFlatParts; ++i) {
        if (v[i].x > 0.f) {
            const float d = v[i].y / v[i].x - pivot;
            s1 += v[i].y;
            q += fmaf(v[i].x * d, d, v[i].z);
        }
    }
    s_red[w][lane] = make_float2(s1, q);
    __syncthreads();
    if (w != 0 || !act) return;
    float t = 0.f, m2 = 0.f;
#pragma unroll
    for (int i = 0; i < kFinWarps; ++i) { t += s_red[i][lane].x; m2 += s_red[i][lane].y; }
    float mean, var;
    merged_stats(N, t, m2, pivot, mean, var);
    put_stats(o, mean, 1.f / sqrtf(var + eps), var, N, momentum, mean_out, invstd_out, running_mean, running_var);
}

// Per-channel constants of the forward apply step and of the backward kernels, loaded (or, in the
// channel-per-CTA kernels, computed) once and passed by value.
struct FwdChan { float mu, is, ga, be, mur, isr, gar, ber; };
struct BwdChan { float mu, is, ga, be, mur, isr; float4 cf, cr; };

// Forward apply of eight frames from t0 on of row (b, o): y = [t < len] * act(gamma * vhat + beta, r).
template <typename T, typename NT>
__device__ __forceinline__ void apply_chunk(const ApplyArgs& a, size_t off, int t0, int len, bool vec, const FwdChan& c) {
    const int Tp = a.Tp;
    float out[8];
    if (t0 < len) {
        float f[8], r[8];
        load_chunk((const NT*)a.v + off, t0, Tp, vec, f);
        if (a.residual == 1) load_chunk((const T*)a.xres + off, t0, Tp, vec, r);
        else if (a.residual == 2) {
            load_chunk((const NT*)a.vr + off, t0, Tp, vec, r);
#pragma unroll
            for (int i = 0; i < 8; ++i) r[i] = fmaf(c.gar, bn_norm(r[i], c.mur, c.isr), c.ber);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) r[i] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float bn = fmaf(c.ga, bn_norm(f[i], c.mu, c.is), c.be);   // the backward pass recomputes exactly this
            float q;
            if (a.res_before_relu) { q = bn + r[i]; if (a.has_relu) q = fmaxf(q, 0.f); }
            else { q = (a.has_relu ? fmaxf(bn, 0.f) : bn) + r[i]; }
            out[i] = (t0 + i < len) ? q : 0.f;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) out[i] = 0.f;
    }
    store_chunk((T*)a.y + off, t0, Tp, vec, out);
}

template <typename T, typename NT>
__global__ void __launch_bounds__(kRowThreads) bn_apply_kernel(ApplyArgs a) {
    pdl_sync();
    SC_ROW_SETUP(a.B * a.C)
    const int b = row / a.C, o = row % a.C, len = min(a.len_out[b], a.Tp);
    FwdChan c{a.mean[o], a.invstd[o], a.gamma[o], a.beta[o], 0.f, 0.f, 0.f, 0.f};
    if (a.residual == 2) { c.mur = a.mean_r[o]; c.isr = a.invstd_r[o]; c.gar = a.gamma_r[o]; c.ber = a.beta_r[o]; }
    for (int t0 = lane * 8; t0 < a.Tp; t0 += 256) apply_chunk<T, NT>(a, (size_t)row * a.Tp, t0, len, a.Tp % 8 == 0, c);
}

// ---- one CTA per channel of a small float32 tensor ---------------------------------------------------------
// In a channel of few eight-frame chunks, what is left of the three steps (row partials, finalize, apply; in the backward
// pass too) is the latency of their launches, about 2.2 us each in a chain of dependent kernels.  One CTA sees the whole
// channel and does all three; the second and third reading of its rows hit the L1 cache.  A block forward and backward:
// 64 channels of 2 x 128 frames 35.9 -> 29.7 us, 128 channels of 7 x 228 frames 75.6 -> 69.7 us.  Against it stand the three
// passes of one CTA where the row-mapped kernels give every (sample, channel) row a warp, and rows that are no whole number
// of chunks, whose elements are loaded one by one in each pass.  Time with the row-mapped kernels over time with this one, 32 to
// 512 channels (blocks without a depthwise step):
//                   chunks   64-256       512          1024         2048
//   whole chunks,  2 samples 1.15-1.44    1.18-1.58    1.14-1.65    1.26-1.70     (256 channels, identity residual: 0.90-1.08)
//                  8 samples 0.95-1.28    1.03-1.19    1.02-1.12    1.01-1.03
//                 32 samples 1.11-1.57    1.04-1.22    0.99-1.05    0.91-1.00
//   other rows (up to 256 channels),
//                  4 samples 0.93-1.41    1.03-1.32    1.04-1.38    1.05-1.40
//                  8 samples 0.97-1.36    1.00-1.19    0.94-1.10    0.96-0.99     (512 channels, 64 / 128 / 256 chunks: 1.23 / 1.02 / 0.87)
//                 16 samples 0.98-1.36    0.89-1.01    0.85-0.98    0.83-0.98     (512 channels: 1.40 / 0.88 / 0.83)
//                 32 samples 1.00-1.33    0.86-1.05    0.84-0.97    0.77-0.88     (512 channels: 1.30 / 1.15 / 1.12)
constexpr int kSmallChunks = 1024, kSmallOddChunks = 256, kSmallOddWork = 256 * 256, kSmallOddSamples = 8;
struct ChanRows {            // chunk j of the channel -> sample and frame
    int cpr, n;
    __device__ __forceinline__ ChanRows(int B, int Tp) : cpr((Tp + 7) >> 3), n(B * ((Tp + 7) >> 3)) {}
    __device__ __forceinline__ void at(int j, int& b, int& t0) const { b = j / cpr; t0 = (j - b * cpr) * 8; }
};
template <int N>
__device__ __forceinline__ void cta_sum(float (&v)[N], float* s_red) {      // in every thread, in warp order
    block_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int i = 0; i < N; ++i) s_red[(threadIdx.x >> 5) * N + i] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[i] = 0.f;
#pragma unroll
        for (int w = 0; w < kRowThreads / 32; ++w) v[i] += s_red[w * N + i];
    }
}

__global__ void __launch_bounds__(kRowThreads)
bn_small_fwd_kernel(ApplyArgs a, const int* __restrict__ nvalid, float eps, float momentum, float* mean_out, float* invstd_out,
                    float* running_mean, float* running_var) {
    __shared__ float s_red[kRowThreads / 32];
    const int o = blockIdx.x, tid = threadIdx.x;
    const ChanRows R(a.B, a.Tp);
    const bool vec = a.Tp % 8 == 0;
    const float N = (float)(*nvalid);
    FwdChan c{0.f, 0.f, a.gamma[o], a.beta[o], 0.f, 0.f, 0.f, 0.f};
    pdl_sync();              // launch_early: the parameters and the count above were settled before the previous kernel
    if (a.residual == 2) { c.mur = a.mean_r[o]; c.isr = a.invstd_r[o]; c.gar = a.gamma_r[o]; c.ber = a.beta_r[o]; }
    float s[1];
    for (int pass = 0; pass < 2; ++pass) {      // the sum, then the squares about the mean
        s[0] = 0.f;
        for (int j = tid; j < R.n; j += kRowThreads) {
            int b, t0;
            R.at(j, b, t0);
            const int len = min(a.len_out[b], a.Tp);
            if (t0 >= len) continue;
            float f[8];
            load_chunk((const float*)a.v + ((size_t)b * a.C + o) * a.Tp, t0, a.Tp, vec, f);
#pragma unroll
            for (int i = 0; i < 8; ++i) if (t0 + i < len) s[0] += pass ? (f[i] - c.mu) * (f[i] - c.mu) : f[i];
        }
        cta_sum(s, s_red);
        if (!pass) c.mu = N > 0.f ? s[0] / N : 0.f;
    }
    const float var = N > 0.f ? s[0] / N : 0.f;
    c.is = 1.f / sqrtf(var + eps);
    if (tid == 0) {
        mean_out[o] = c.mu; invstd_out[o] = c.is;
        if (running_mean) running_mean[o] = (1.f - momentum) * running_mean[o] + momentum * c.mu;
        if (running_var) running_var[o] = (1.f - momentum) * running_var[o] + momentum * (N > 1.f ? var * (N / (N - 1.f)) : var);
    }
    for (int j = tid; j < R.n; j += kRowThreads) {
        int b, t0;
        R.at(j, b, t0);
        apply_chunk<float, float>(a, ((size_t)b * a.C + o) * a.Tp, t0, min(a.len_out[b], a.Tp), vec, c);
    }
}

// Shared by the reduce and apply steps of the backward pass: per element gate and normalised value.
template <typename T, typename NT>
struct BwdRow {
    const T* __restrict__ g; const T* __restrict__ y; const NT* __restrict__ v; const NT* __restrict__ vr;
    float gam, bet, mu, is, mur, isr;
    int len, Tp;
    bool vec;
    __device__ BwdRow(const BnBwdArgs& a, int row, int b, int o) {
        Tp = a.Tp; len = min(a.len_out[b], Tp); vec = (Tp % 8 == 0);
        g = (const T*)a.g + (size_t)row * Tp;
        y = a.y ? (const T*)a.y + (size_t)row * Tp : nullptr;
        v = a.has_bn ? (const NT*)a.v + (size_t)row * Tp : nullptr;
        vr = (a.residual == 2) ? (const NT*)a.vr + (size_t)row * Tp : nullptr;
        const bool own_gate = a.has_relu && !a.res_before_relu && a.has_bn;
        gam = own_gate ? a.gamma[o] : 1.f; bet = own_gate ? a.beta[o] : 0.f;
        mu = a.has_bn ? a.mean[o] : 0.f; is = a.has_bn ? a.invstd[o] : 0.f;
        mur = (a.residual == 2) ? a.mean_r[o] : 0.f; isr = (a.residual == 2) ? a.invstd_r[o] : 0.f;
    }
    // ga: gated upstream gradient; gr: gradient reaching the residual sum; vn/vnr: normalised values
    __device__ __forceinline__ void chunk(const BnBwdArgs& a, int t0, float (&ga)[8], float (&gr)[8],
                                          float (&vn)[8], float (&vnr)[8]) const {
        float fg[8], fy[8];
        load_chunk(g, t0, Tp, vec, fg);
        const bool need_y = a.has_relu && a.res_before_relu;
        if (need_y) load_chunk(y, t0, Tp, vec, fy);
        if (a.has_bn) {
            load_chunk(v, t0, Tp, vec, vn);
#pragma unroll
            for (int i = 0; i < 8; ++i) vn[i] = bn_norm(vn[i], mu, is);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) vn[i] = 0.f;
        }
        if (a.residual == 2) {
            load_chunk(vr, t0, Tp, vec, vnr);
#pragma unroll
            for (int i = 0; i < 8; ++i) vnr[i] = bn_norm(vnr[i], mur, isr);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) vnr[i] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const bool in = (t0 + i < len);
            const float gm = in ? fg[i] : 0.f;
            bool gate = true;
            if (a.has_relu) gate = a.res_before_relu ? (fy[i] > 0.f) : (fmaf(gam, vn[i], bet) > 0.f);
            ga[i] = gate ? gm : 0.f;
            gr[i] = a.res_before_relu ? ga[i] : gm;
            if (!in) { vn[i] = 0.f; vnr[i] = 0.f; }
        }
    }
};

// Partial sums of the backward reduction live in a [sample][slot][channel] array, so that the finalize
// kernel, which gives one channel to each lane, reads contiguous runs.
__device__ __forceinline__ size_t bwd_part_index(const BnBwdArgs& a, int b, int slot, int o) {
    return ((size_t)b * a.nslots + slot) * a.C + o;
}

template <typename T, typename NT>
__global__ void __launch_bounds__(kRowThreads) bn_bwd_reduce_kernel(BnBwdArgs a) {
    pdl_sync();
    SC_ROW_SETUP(a.B * a.C)
    const int b = row / a.C, o = row % a.C;
    BwdRow<T, NT> R(a, row, b, o);
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    float amax = 0.f;
    for (int t0 = lane * 8; t0 < R.len; t0 += 256) {
        float ga[8], gr[8], vh[8], vhr[8];
        R.chunk(a, t0, ga, gr, vh, vhr);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            s[0] += ga[i]; s[1] += ga[i] * vh[i]; s[2] += gr[i]; s[3] += gr[i] * vhr[i];
            amax = fmaxf(amax, fmaxf(fabsf(ga[i]), fabsf(gr[i])));
        }
    }
    block_sum(s);
    if (a.gmax) amax = block_max(amax);
    if (lane == 0) {
        a.partials[bwd_part_index(a, b, 0, o)] = make_float4(s[0], s[1], s[2], s[3]);
        if (a.gmax) a.amax_part[bwd_part_index(a, b, 0, o)] = amax;
    }
}

// What the sums of channel o over all frames amount to: the coefficients of the apply step (cf, cr), the channel's parameter
// gradients (one thread writes them) and its term of the bound on |gv|.
struct BwdGrads { const float *gamma, *gamma_r; float *dgamma, *dbeta, *dgamma_r, *dbeta_r, *dbias; int accumulate; };
__device__ __forceinline__ void bwd_channel(const BnBwdArgs& a, const BwdGrads& p, int o, bool writes, float d0, float d1, float d2,
                                            float d3, float amax, float4& cf, float4& cr) {
    const float N = (float)(*a.nvalid);
    if (a.gmax && writes) {
        // |gv| <= |k| (max|ga| + |c1| + max|vhat| |c2|) and max|vhat| <= sqrt(N); a maximum is order-free,
        // so the integer atomic on the (non-negative) float's bit pattern keeps the result repeatable
        float bound = amax;
        if (a.has_bn)
            bound = fabsf(p.gamma[o] * a.invstd[o]) * (amax + fabsf(d0) / N + sqrtf(N) * fabsf(d1) / N);
        if (a.residual == 2)     // the residual branch's gradient shares the scale
            bound = fmaxf(bound, fabsf(p.gamma_r[o] * a.invstd_r[o]) *
                                     (amax + fabsf(d2) / N + sqrtf(N) * fabsf(d3) / N));
        if (bound < 3.0e38f) atomicMax(reinterpret_cast<unsigned int*>(a.gmax), __float_as_uint(bound));
    }
    auto put = [&](float* dst, float val) {
        if (dst && writes) dst[o] = p.accumulate ? dst[o] + val : val;
    };
    if (a.has_bn) {
        put(p.dbeta, d0); put(p.dgamma, d1);
        cf = make_float4(p.gamma[o] * a.invstd[o], d0 / N, d1 / N, 0.f);
    } else {
        put(p.dbias, d0);
        cf = make_float4(1.f, 0.f, 0.f, 0.f);
    }
    if (a.residual == 2) {
        put(p.dbeta_r, d2); put(p.dgamma_r, d3);
        cr = make_float4(p.gamma_r[o] * a.invstd_r[o], d2 / N, d3 / N, 0.f);
    }
}

// Thirty-two channels per CTA, one per lane; warp w takes samples w, w + 32, ... with all their slots (every
// load issued before the first add) and the thirty-two warp results are combined in warp order
// (bit-repeatable).
constexpr int kBwdMaxSlotsUnrolled = 8;
constexpr int kRedV = 2, kRedVectors = 32 * kRedV;       // vectors per lane and per warp of the flattened reduction
__global__ void __launch_bounds__(32 * kFinWarps)
bn_bwd_finalize_kernel(BnBwdArgs a, BwdGrads p) {
    pdl_sync();
    __shared__ float4 s_sum[kFinWarps][32];
    __shared__ float s_max[kFinWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    const bool act = o < a.C;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, amax = 0.f;
    if (act) {
        const uint32_t vpr = (uint32_t)(a.Tp / 8);
        for (int b = w; b < a.B; b += kFinWarps) {
            int used = 1;
            if (a.nslots > 1) {      // slots in use for this row (see bn_bwd_reduce_fast_kernel); r * vpr < 2^31
                const uint32_t r = (uint32_t)b * (uint32_t)a.C + (uint32_t)o;
                used = (int)(((r + 1u) * vpr - 1u) / kRedVectors - (r * vpr) / kRedVectors) + 1;
            }
            for (int sl0 = 0; sl0 < used; sl0 += kBwdMaxSlotsUnrolled) {
                float4 pv[kBwdMaxSlotsUnrolled]; float am[kBwdMaxSlotsUnrolled];
#pragma unroll
                for (int i = 0; i < kBwdMaxSlotsUnrolled; ++i) {
                    const bool use = sl0 + i < used;
                    pv[i] = use ? a.partials[bwd_part_index(a, b, sl0 + i, o)] : make_float4(0.f, 0.f, 0.f, 0.f);
                    am[i] = (use && a.gmax) ? a.amax_part[bwd_part_index(a, b, sl0 + i, o)] : 0.f;
                }
#pragma unroll
                for (int i = 0; i < kBwdMaxSlotsUnrolled; ++i) {
                    s0 += pv[i].x; s1 += pv[i].y; s2 += pv[i].z; s3 += pv[i].w;
                    amax = fmaxf(amax, am[i]);
                }
            }
        }
    }
    s_sum[w][lane] = make_float4(s0, s1, s2, s3);
    s_max[w][lane] = amax;
    __syncthreads();
    if (w != 0 || !act) return;
    float d0 = 0.f, d1 = 0.f, d2 = 0.f, d3 = 0.f;
    amax = 0.f;
#pragma unroll
    for (int i = 0; i < kFinWarps; ++i) {
        const float4 q = s_sum[i][lane];
        d0 += q.x; d1 += q.y; d2 += q.z; d3 += q.w;
        amax = fmaxf(amax, s_max[i][lane]);
    }
    float4 cf, cr = make_float4(0.f, 0.f, 0.f, 0.f);
    bwd_channel(a, p, o, true, d0, d1, d2, d3, amax, cf, cr);
    a.coef[o] = cf;
    if (a.residual == 2) a.coef_r[o] = cr;
}

// Backward apply of eight frames from t0 on of the row that R describes (cf, cr: the channel's coefficients).
template <typename T, typename NT, typename GT>
__device__ __forceinline__ void bwd_apply_chunk(const BnBwdArgs& a, const BwdRow<T, NT>& R, size_t off, int t0, const float4& cf,
                                                const float4& cr, float sc) {
    float o1[8], o2[8];
    if (t0 < R.len) {
        float ga[8], gr[8], vh[8], vhr[8];
        R.chunk(a, t0, ga, gr, vh, vhr);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const bool in = (t0 + i < R.len);
            o1[i] = in ? cf.x * (ga[i] - cf.y - vh[i] * cf.z) : 0.f;
            if (a.residual == 2) o2[i] = in ? cr.x * (gr[i] - cr.y - vhr[i] * cr.z) : 0.f;
            else o2[i] = gr[i];
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) { o1[i] = 0.f; o2[i] = 0.f; }
    }
    const int nin = R.len - t0;
    if (a.gv16) {              // half copy for the weight gradient; gv itself keeps plain rounding
        float h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = o1[i] * sc;
        diffuse8<__half>(h, nin);
        store_chunk((__half*)a.gv16 + off, t0, R.Tp, R.vec, h);
    } else {
        if (a.gv_scaled) {
#pragma unroll
            for (int i = 0; i < 8; ++i) o1[i] *= sc;
        }
        diffuse8<GT>(o1, nin);
    }
    if (a.gvr16) {
        float h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = o2[i] * sc;
        diffuse8<__half>(h, nin);
        store_chunk((__half*)a.gvr16 + off, t0, R.Tp, R.vec, h);
    } else if (a.residual == 2) {
        diffuse8<T>(o2, nin);
    }
    store_chunk((GT*)a.gv + off, t0, R.Tp, R.vec, o1);
    if (a.residual == 2) store_chunk((T*)a.gvr + off, t0, R.Tp, R.vec, o2);
    if (a.residual == 1) store_chunk((T*)a.gres + off, t0, R.Tp, R.vec, o2);
}

template <typename T, typename NT, typename GT>
__global__ void __launch_bounds__(kRowThreads) bn_bwd_apply_kernel(BnBwdArgs a) {
    pdl_sync();
    SC_ROW_SETUP(a.B * a.C)
    const int b = row / a.C, o = row % a.C;
    BwdRow<T, NT> R(a, row, b, o);
    const float4 cf = a.coef[o];
    const float sc = a.gmax ? pow2_scale(*a.gmax) : 1.f;      // multiplying by it is exact: a power of two
    const float4 cr = (a.residual == 2) ? a.coef_r[o] : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int t0 = lane * 8; t0 < R.Tp; t0 += 256) bwd_apply_chunk<T, NT, GT>(a, R, (size_t)row * R.Tp, t0, cf, cr, sc);
}

// The backward counterpart of bn_small_fwd_kernel.
__global__ void __launch_bounds__(kRowThreads) bn_small_bwd_kernel(BnBwdArgs a, BwdGrads p) {
    pdl_sync();
    __shared__ float s_red[4 * kRowThreads / 32];
    const int o = blockIdx.x, tid = threadIdx.x;
    const ChanRows C(a.B, a.Tp);
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int j = tid; j < C.n; j += kRowThreads) {
        int b, t0;
        C.at(j, b, t0);
        const BwdRow<float, float> R(a, b * a.C + o, b, o);
        if (t0 >= R.len) continue;
        float ga[8], gr[8], vh[8], vhr[8];
        R.chunk(a, t0, ga, gr, vh, vhr);
#pragma unroll
        for (int i = 0; i < 8; ++i) { s[0] += ga[i]; s[1] += ga[i] * vh[i]; s[2] += gr[i]; s[3] += gr[i] * vhr[i]; }
    }
    cta_sum(s, s_red);
    float4 cf, cr = make_float4(0.f, 0.f, 0.f, 0.f);
    bwd_channel(a, p, o, tid == 0, s[0], s[1], s[2], s[3], 0.f, cf, cr);
    for (int j = tid; j < C.n; j += kRowThreads) {
        int b, t0;
        C.at(j, b, t0);
        const int row = b * a.C + o;
        bwd_apply_chunk<float, float, float>(a, BwdRow<float, float>(a, row, b, o), (size_t)row * a.Tp, t0, cf, cr, 1.f);
    }
}

// One 8-frame vector of the forward apply step: y = [t < len] * relu(gamma * vhat + beta (+ r)); n = frames of the
// vector inside the sample (0: wholly padding), rv / rr = the raw 16 bytes of v and of the residual operand.
template <typename T, typename NT, int RES>
__device__ __forceinline__ void apply_core(T* yp, int n, const uint4& rv, const uint4& rr, const FwdChan& c) {
    float out[8];
    if (n > 0) {
        float f[8], r[8];
        cvt8<NT>(rv, f);
        if (RES == 1) cvt8<T>(rr, r);
        if (RES == 2) cvt8<NT>(rr, r);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float rres = 0.f;
            if (RES == 1) rres = r[i];
            if (RES == 2) rres = fmaf(c.gar, bn_norm(r[i], c.mur, c.isr), c.ber);
            const float q = fmaxf(fmaf(c.ga, bn_norm(f[i], c.mu, c.is), c.be) + rres, 0.f);
            out[i] = i < n ? q : 0.f;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) out[i] = 0.f;
    }
    st8<T>(yp, out);
}
template <int RES> __device__ __forceinline__ void fwd_chan(const ApplyArgs& a, int o, FwdChan& c) {
    c.mu = a.mean[o]; c.is = a.invstd[o]; c.ga = a.gamma[o]; c.be = a.beta[o];
    if (RES == 2) { c.mur = a.mean_r[o]; c.isr = a.invstd_r[o]; c.gar = a.gamma_r[o]; c.ber = a.beta_r[o]; }
}
template <typename T, typename NT, int RES>
__device__ __forceinline__ void apply_vec(const ApplyArgs& a, int o, int n, size_t off, const uint4& rv, const uint4& rr) {
    FwdChan c{};
    if (n > 0) fwd_chan<RES>(a, o, c);
    apply_core<T, NT, RES>((T*)a.y + off, n, rv, rr, c);
}

// One 8-frame vector of the backward apply step (gv and the residual branch's gradient), computed and stored.
template <typename T, typename NT, typename GT, int RES>
__device__ __forceinline__ void bwd_apply_core(const BnBwdArgs& a, int n, size_t off, float sc, bool fold, const uint4& rg,
                                               const uint4& rv, const uint4& rr, const uint4& ry, const BwdChan& c) {
    float o1[8], o2[8];
    if (n > 0) {
        float g[8], y[8], vn[8], vnr[8];
        cvt8<T>(rg, g);
        cvt8<NT>(rv, vn);
        const uint64_t nmu2 = pk::pack(-c.mu, -c.mu), is2 = pk::pack(c.is, c.is);
        uint64_t vn2[4], vr2[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) vn2[q] = pk::bn_norm2(pk::pack(vn[2 * q], vn[2 * q + 1]), nmu2, is2);
        if (RES == 2) {
            cvt8<NT>(rr, vnr);
            const uint64_t nmur2 = pk::pack(-c.mur, -c.mur), isr2 = pk::pack(c.isr, c.isr);
#pragma unroll
            for (int q = 0; q < 4; ++q) vr2[q] = pk::bn_norm2(pk::pack(vnr[2 * q], vnr[2 * q + 1]), nmur2, isr2);
        }
        bool gate[8];
        if (RES == 0) {
            // without a residual the forward output is relu(gamma * vhat + beta), rounded to the
            // activation type: the gate is recomputed from v and the output need not be read
            const uint64_t ga2 = pk::pack(c.ga, c.ga), be2 = pk::pack(c.be, c.be);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float a0, a1;
                pk::unpack(pk::fma(ga2, vn2[q], be2), a0, a1);
                gate[2 * q] = rounds_positive<T>(a0); gate[2 * q + 1] = rounds_positive<T>(a1);
            }
        } else {
            cvt8<T>(ry, y);
#pragma unroll
            for (int i = 0; i < 8; ++i) gate[i] = y[i] > 0.f;
        }
        // gv = k (ga - c1 - c2 vhat) as two fused multiply-adds; when gv itself is the scaled half tensor the
        // power-of-two scale is folded into k (exact)
        const float4 cf = c.cf;
        const float kx = (fold ? sc : 1.f) * cf.x;
        const uint64_t kx2 = pk::pack(kx, kx), k02 = pk::pack(-kx * cf.y, -kx * cf.y), k22 = pk::pack(-kx * cf.z, -kx * cf.z);
        uint64_t kr2 = 0, r02 = 0, r22 = 0;
        if (RES == 2) {
            const float4 cr = c.cr;
            kr2 = pk::pack(cr.x, cr.x); r02 = pk::pack(-cr.x * cr.y, -cr.x * cr.y); r22 = pk::pack(-cr.x * cr.z, -cr.x * cr.z);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool in0 = 2 * q < n, in1 = 2 * q + 1 < n;
            const float g0 = (in0 && gate[2 * q]) ? g[2 * q] : 0.f;
            const float g1 = (in1 && gate[2 * q + 1]) ? g[2 * q + 1] : 0.f;
            const uint64_t ga2 = pk::pack(g0, g1);
            float x0, x1;
            pk::unpack(pk::fma(k22, vn2[q], pk::fma(kx2, ga2, k02)), x0, x1);
            o1[2 * q] = in0 ? x0 : 0.f; o1[2 * q + 1] = in1 ? x1 : 0.f;
            if (RES == 2) {
                pk::unpack(pk::fma(r22, vr2[q], pk::fma(kr2, ga2, r02)), x0, x1);
                o2[2 * q] = in0 ? x0 : 0.f; o2[2 * q + 1] = in1 ? x1 : 0.f;
            }
            if (RES == 1) { o2[2 * q] = g0; o2[2 * q + 1] = g1; }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) { o1[i] = 0.f; o2[i] = 0.f; }
    }
    if (a.gv16) {            // half copy for the weight gradient; gv itself keeps plain rounding
        float h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = o1[i] * sc;
        diffuse8<__half>(h, n);
        st8<__half>((__half*)a.gv16 + off, h);
    } else {
        diffuse8<GT>(o1, n);
    }
    if (RES == 2) {
        if (a.gvr16) {
            float h[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) h[i] = o2[i] * sc;
            diffuse8<__half>(h, n);
            st8<__half>((__half*)a.gvr16 + off, h);
        } else {
            diffuse8<T>(o2, n);
        }
    }
    st8<GT>((GT*)a.gv + off, o1);
    if (RES == 2) st8<T>((T*)a.gvr + off, o2);
    if (RES == 1) st8<T>((T*)a.gres + off, o2);
}

template <typename T, typename NT, typename GT, int RES>
__device__ __forceinline__ void bwd_apply_vec(const BnBwdArgs& a, int o, int n, size_t off, float sc, bool fold,
                                              const uint4& rg, const uint4& rv, const uint4& rr, const uint4& ry) {
    BwdChan c{};
    if (n > 0) {
        c.mu = a.mean[o]; c.is = a.invstd[o]; c.cf = a.coef[o];
        if (RES == 0) { c.ga = a.gamma[o]; c.be = a.beta[o]; }
        if (RES == 2) { c.mur = a.mean_r[o]; c.isr = a.invstd_r[o]; c.cr = a.coef_r[o]; }
    }
    bwd_apply_core<T, NT, GT, RES>(a, n, off, sc, fold, rg, rv, rr, ry, c);
}

// One 8-frame vector of the backward reduction: s0 = sum ga, s1 = sum ga * vhat, s3 = sum ga * vhat_r, m = max |ga|
// over its n (> 0) frames inside the sample.
template <typename T, typename NT, int RES>
__device__ __forceinline__ void reduce_core(int n, const uint4& rg, const uint4& rv, const uint4& rr, const uint4& ry,
                                            const BwdChan& c, float& s0, float& s1, float& s3, float& m_out) {
    float g[8], y[8], vn[8], vnr[8];
    cvt8<T>(rg, g);
    cvt8<NT>(rv, vn);
    const uint64_t nmu2 = pk::pack(-c.mu, -c.mu), is2 = pk::pack(c.is, c.is);
    uint64_t vn2[4], vr2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) vn2[q] = pk::bn_norm2(pk::pack(vn[2 * q], vn[2 * q + 1]), nmu2, is2);
    if (RES == 2) {
        cvt8<NT>(rr, vnr);
        const uint64_t nmur2 = pk::pack(-c.mur, -c.mur), isr2 = pk::pack(c.isr, c.isr);
#pragma unroll
        for (int q = 0; q < 4; ++q) vr2[q] = pk::bn_norm2(pk::pack(vnr[2 * q], vnr[2 * q + 1]), nmur2, isr2);
    }
    bool gate[8];
    if (RES == 0) {          // gate from v (see bn_bwd_apply_fast_kernel)
        const uint64_t ga2 = pk::pack(c.ga, c.ga), be2 = pk::pack(c.be, c.be);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float a0, a1;
            pk::unpack(pk::fma(ga2, vn2[q], be2), a0, a1);
            gate[2 * q] = rounds_positive<T>(a0); gate[2 * q + 1] = rounds_positive<T>(a1);
        }
    } else {
        cvt8<T>(ry, y);
#pragma unroll
        for (int i = 0; i < 8; ++i) gate[i] = y[i] > 0.f;
    }
    uint64_t s0_2 = pk::pack(0.f, 0.f), s1_2 = pk::pack(0.f, 0.f), s3_2 = pk::pack(0.f, 0.f);
    float m = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float g0 = (2 * q < n && gate[2 * q]) ? g[2 * q] : 0.f;
        const float g1 = (2 * q + 1 < n && gate[2 * q + 1]) ? g[2 * q + 1] : 0.f;
        const uint64_t ga2 = pk::pack(g0, g1);
        s0_2 = pk::add(s0_2, ga2);
        s1_2 = pk::fma(ga2, vn2[q], s1_2);
        if (RES == 2) s3_2 = pk::fma(ga2, vr2[q], s3_2);
        m = fmaxf(m, fmaxf(fabsf(g0), fabsf(g1)));
    }
    float t0_, t1_;
    pk::unpack(s0_2, t0_, t1_); s0 = t0_ + t1_;
    pk::unpack(s1_2, t0_, t1_); s1 = t0_ + t1_;
    pk::unpack(s3_2, t0_, t1_); s3 = t0_ + t1_;
    m_out = m;
}

template <typename T, typename NT, int RES>
__device__ __forceinline__ void reduce_vec(const BnBwdArgs& a, int o, int n, const uint4& rg, const uint4& rv, const uint4& rr,
                                           const uint4& ry, float& s0, float& s1, float& s3, float& m_out) {
    BwdChan c{};
    c.mu = a.mean[o]; c.is = a.invstd[o];
    if (RES == 0) { c.ga = a.gamma[o]; c.be = a.beta[o]; }
    if (RES == 2) { c.mur = a.mean_r[o]; c.isr = a.invstd_r[o]; }
    reduce_core<T, NT, RES>(n, rg, rv, rr, ry, c, s0, s1, s3, m_out);
}

// ---- flattened fast paths (the encoder's configuration: BN + ReLU, residual joined before the ReLU,
// rows a multiple of 8 frames).  A warp takes 32 * V consecutive 8-frame vectors, lane l the vectors
// l, l + 32, ...: no row tails, and V independent 16-byte loads per tensor in flight per thread.
template <typename T, typename NT, int RES, int V>
__global__ void __launch_bounds__(256) bn_apply_fast_kernel(ApplyArgs a, int vpr, long long total) {
    const uint32_t tid = blockIdx.x * 256u + threadIdx.x;        // the launcher guarantees total < 2^31
    const uint32_t base = (tid >> 5) * (32u * V) + (threadIdx.x & 31), tot = (uint32_t)total;
    size_t off[V]; int nin[V], ch[V];
    uint4 rv[V], rr[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const uint32_t idx = base + 32u * j;
        nin[j] = -1; ch[j] = 0; off[j] = 0;
        rv[j] = make_uint4(0, 0, 0, 0); rr[j] = make_uint4(0, 0, 0, 0);
        if (idx < tot) {
            const int row = (int)a.dvpr.div(idx), t0 = ((int)idx - row * vpr) * 8;
            const int b = (int)a.dC.div((uint32_t)row);
            ch[j] = row - b * a.C;
            nin[j] = max(0, min(a.len_out[b], a.Tp) - t0);
            off[j] = (size_t)row * a.Tp + t0;
        }
    }
    pdl_sync();              // indices and lengths are worked out ahead of the wait (launch_early)
#pragma unroll
    for (int j = 0; j < V; ++j) {
        if (nin[j] > 0) {
            rv[j] = *reinterpret_cast<const uint4*>((const NT*)a.v + off[j]);
            if (RES == 1) rr[j] = *reinterpret_cast<const uint4*>((const T*)a.xres + off[j]);
            if (RES == 2) rr[j] = *reinterpret_cast<const uint4*>((const NT*)a.vr + off[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < V; ++j) {
        if (nin[j] < 0) continue;
        apply_vec<T, NT, RES>(a, ch[j], nin[j], off[j], rv[j], rr[j]);
    }
}

// The same step from packed v / vr to dense y: a thread takes one aligned 8-element vector of the dense tensor and gathers the
// packed operands (two vectors per thread took 30.0 us where one takes 26.1, bf16, 23 x 384 x 797, projected residual: registers
// against warps in flight).  A vector that runs over the end of a row (of at least 8 frames) is spliced from this row's last
// frames and the next row's first; shorter rows are done element by element.  Blocks past the tensor's own copy u out.
// What it replaces: four extra passes (v, vr, y and u copied to dense form one after the other) and their launches.
template <typename T, typename NT, int RES, int D>
__global__ void __launch_bounds__(256) bn_apply_unpack_kernel(ApplyArgs a, uint32_t total, int nblk_apply, uint32_t total_u) {
    const bool copy = (int)blockIdx.x >= nblk_apply;
    const int C = copy ? a.Cu : a.C, nrows = a.B * C;
    const uint32_t tot = copy ? total_u : total;
    const uint32_t tot_packed = (uint32_t)a.B * D * C * a.Tp;
    const bool aligned = (a.T & 7) == 0, vector_rows = a.T >= 8;
    const uint32_t f = ((blockIdx.x - (copy ? nblk_apply : 0)) * 256u + threadIdx.x) * 8u;      // first element
    int row = 0, t = 0, b = 0, ch = 0, n = 0;
    if (f < tot) {
        row = (int)a.dT.div(f); t = (int)(f - (uint32_t)row * a.T);
        b = row / C; ch = row - b * C;
        n = min(a.len_out[b], a.T) - t;
    }
    pdl_sync();              // the lengths above: launch_early
    if (f >= tot) return;
    const int left = (int)min(8u, tot - f);
    if (vector_rows) {
        Packed8<D> rv, rr; uint4 rx = make_uint4(0, 0, 0, 0);
        if (n > 0) {
            rv = Packed8<D>(copy ? a.u : a.v, b, ch, C, a.Tp, t, tot_packed, aligned);
            if (RES == 2 && !copy) rr = Packed8<D>(a.vr, b, ch, C, a.Tp, t, tot_packed, aligned);
        }
        // the dense operand is aligned like the result (the last vector may hold less than eight elements)
        if (RES == 1 && !copy) rx = fetch<1>(a.xres, f, tot).v[0];
        uint4 q = rv.get(), qr = RES == 2 ? rr.get() : rx, y = make_uint4(0, 0, 0, 0);
        if (!copy) {
            FwdChan c{};
            fwd_chan<RES>(a, ch, c);
            apply_core<T, NT, RES>((T*)&y, n, q, qr, c);
        } else if (n < 8) q = keep_first(q, n);
        const int k = a.T - t;                                 // elements of this row
        if (k < 8 && row + 1 < nrows) {
            const int b2 = (row + 1) / C, c2 = row + 1 - b2 * C, n2 = min(a.len_out[b2], a.T) + k;
            uint4 p = Packed8<D>(copy ? a.u : a.v, b2, c2, C, a.Tp, -k, tot_packed, false).get(), pr = rx, y2;
            if (RES == 2 && !copy) pr = Packed8<D>(a.vr, b2, c2, C, a.Tp, -k, tot_packed, false).get();
            if (!copy) {
                FwdChan c{};
                fwd_chan<RES>(a, c2, c);
                apply_core<T, NT, RES>((T*)&y2, n2, p, pr, c);
                y = splice(y, y2, k);
            } else if (n2 < 8) p = keep_first(p, n2);
            q = splice(q, p, k);
            if (RES == 2) qr = splice(qr, pr, k);
        }
        if (copy) { st8_first((unsigned short*)a.u_out + f, q, left); return; }
        st8_first((unsigned short*)a.y + f, y, left);
        if (a.v_out) st8_first((unsigned short*)a.v_out + f, q, left);
        if (RES == 2 && a.vr_out) st8_first((unsigned short*)a.vr_out + f, qr, left);
        return;
    }
    for (uint32_t e = f; e < f + left; ++e) {
        const int row_e = (int)a.dT.div(e), te = (int)(e - (uint32_t)row_e * a.T);
        const int be = row_e / C, o = row_e - be * C;
        const bool in = te < min(a.len_out[be], a.T);
        const uint32_t q = D == 1 ? (uint32_t)row_e * a.Tp + te : ((uint32_t)(be * 2 + (te & 1)) * C + o) * a.Tp + (te >> 1);
        if (copy) { ((unsigned short*)a.u_out)[e] = in ? ((const unsigned short*)a.u)[q] : (unsigned short)0; continue; }
        const NT vq = in ? ((const NT*)a.v)[q] : NT(0.f);
        float r = 0.f;
        if (RES == 1 && in) r = ldf((const T*)a.xres + e);
        if (RES == 2) {
            const NT vrq = in ? ((const NT*)a.vr)[q] : NT(0.f);
            r = fmaf(a.gamma_r[o], bn_norm(ldf(&vrq), a.mean_r[o], a.invstd_r[o]), a.beta_r[o]);
            if (a.vr_out) ((NT*)a.vr_out)[e] = vrq;
        }
        const float y = fmaxf(fmaf(a.gamma[o], bn_norm(ldf(&vq), a.mean[o], a.invstd[o]), a.beta[o]) + r, 0.f);
        stf((T*)a.y + e, in ? y : 0.f);
        if (a.v_out) ((NT*)a.v_out)[e] = vq;
    }
}

// Operand of the backward kernels: eight frames of packed row (b, o), position t0 of it, from a tensor that has the same
// (packed) layout (G = 0, element offset off) or is dense with one or two phases per sample (G = 1, 2).  n > 0 frames
// are inside the sample; a dense tensor's frames past them are unspecified and come back as zero (a masked gradient times
// a NaN would not be zero).
template <int G> struct BwdRaw {
    RawVec<G + 1> r; uint32_t idx;
    __device__ __forceinline__ BwdRaw() : r{}, idx(0) {}
    __device__ __forceinline__ BwdRaw(const BnBwdArgs& a, const void* src, size_t off, int b, int o, int t0) : idx(0) {
        if (G == 0) { r.v[0] = *reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned short*>(src) + off); return; }
        idx = G == 1 ? ((uint32_t)b * a.C + o) * a.T + t0 : ((uint32_t)(b >> 1) * a.C + o) * a.T + 2 * t0 + (b & 1);
        r = fetch<G + 1>(src, idx, a.total_dense);
    }
    __device__ __forceinline__ uint4 get(int n) const;
};
template <> __device__ __forceinline__ uint4 BwdRaw<0>::get(int) const { return r.v[0]; }
template <> __device__ __forceinline__ uint4 BwdRaw<1>::get(int n) const { const uint4 q = pick8(r, idx); return n < 8 ? keep_first(q, n) : q; }
template <> __device__ __forceinline__ uint4 BwdRaw<2>::get(int n) const { const uint4 q = pick8_even(r, idx); return n < 8 ? keep_first(q, n) : q; }

template <typename T, typename NT, typename GT, int RES, int V, int G>
__global__ void __launch_bounds__(256) bn_bwd_apply_fast_kernel(BnBwdArgs a, int vpr, long long total) {
    const uint32_t tid = blockIdx.x * 256u + threadIdx.x;        // the launcher guarantees total < 2^31
    const uint32_t base = (tid >> 5) * (32u * V) + (threadIdx.x & 31), tot = (uint32_t)total;
    const bool fold = !a.gv16 && a.gv_scaled;
    size_t off[V]; int nin[V], ch[V], bs[V], t0s[V];
    BwdRaw<G> rg[V], rv[V], rr[V], ry[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const uint32_t idx = base + 32u * j;
        nin[j] = -1; ch[j] = 0; off[j] = 0; bs[j] = 0; t0s[j] = 0;
        if (idx < tot) {
            const int row = (int)a.dvpr.div(idx);
            t0s[j] = ((int)idx - row * vpr) * 8;
            bs[j] = (int)a.dC.div((uint32_t)row);
            ch[j] = row - bs[j] * a.C;
            const int len = min(a.len_out[bs[j]], a.Tp);
            nin[j] = max(0, len - t0s[j]);                                // frames of this vector inside the sample
            // with half of a batch in padding the zeros were a quarter of this kernel's traffic
            if (RES != 1 && a.skip_padding && t0s[j] >= ((len + 63) & ~63)) nin[j] = -1;
            off[j] = (size_t)row * a.Tp + t0s[j];
        }
    }
    pdl_sync();              // as in the forward apply step
    const float sc = a.gmax ? pow2_scale(*a.gmax) : 1.f;          // multiplying by it is exact: a power of two
#pragma unroll
    for (int j = 0; j < V; ++j) {
        if (nin[j] > 0) {
            const int b = bs[j], t0 = t0s[j];
            rg[j] = BwdRaw<G>(a, a.g, off[j], b, ch[j], t0);
            rv[j] = BwdRaw<G>(a, a.v, off[j], b, ch[j], t0);
            if (RES == 2) rr[j] = BwdRaw<G>(a, a.vr, off[j], b, ch[j], t0);
            if (RES != 0) ry[j] = BwdRaw<G>(a, a.y, off[j], b, ch[j], t0);
        }
    }
#pragma unroll
    for (int j = 0; j < V; ++j) {
        if (nin[j] < 0) continue;
        bwd_apply_vec<T, NT, GT, RES>(a, ch[j], nin[j], off[j], sc, fold, rg[j].get(nin[j]), rv[j].get(nin[j]), rr[j].get(nin[j]), ry[j].get(nin[j]));
    }
}

// Flattened reduce: a warp's kRedVectors consecutive vectors belong to at most two rows (vpr >= kRedVectors), so two
// masked warp reductions give one partial per (row, warp) pair.  Row r's partials sit in slots
// [0, last_warp(r) - first_warp(r)] with first_warp(r) = (r * vpr) / kRedVectors: a static assignment,
// summed later in slot order.
template <typename T, typename NT, int RES>
__global__ void __launch_bounds__(256) bn_bwd_reduce_fast_kernel(BnBwdArgs a, int vpr, long long total) {
    pdl_sync();
    constexpr int V = kRedV;
    const uint32_t tid = blockIdx.x * 256u + threadIdx.x;        // the launcher guarantees total < 2^31
    const int lane = threadIdx.x & 31;
    const uint32_t wg = tid >> 5;                                // global warp index
    const uint32_t warp_first = wg * (32u * V), tot = (uint32_t)total;
    if (warp_first >= tot) return;
    const int row0 = (int)a.dvpr.div(warp_first);
    int nin[V], ch[V], rw[V];
    uint4 rg[V], rv[V], rr[V], ry[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const uint32_t idx = warp_first + 32u * j + lane;
        nin[j] = 0; ch[j] = 0; rw[j] = row0;
        rg[j] = rv[j] = rr[j] = ry[j] = make_uint4(0, 0, 0, 0);
        if (idx < tot) {
            const int row = (int)a.dvpr.div(idx), t0 = ((int)idx - row * vpr) * 8;
            const int b = (int)a.dC.div((uint32_t)row);
            rw[j] = row; ch[j] = row - b * a.C;
            nin[j] = max(0, min(a.len_out[b], a.Tp) - t0);
            if (nin[j] > 0) {
                const size_t off = (size_t)row * a.Tp + t0;
                rg[j] = *reinterpret_cast<const uint4*>((const T*)a.g + off);
                rv[j] = *reinterpret_cast<const uint4*>((const NT*)a.v + off);
                if (RES == 2) rr[j] = *reinterpret_cast<const uint4*>((const NT*)a.vr + off);
                if (RES != 0) ry[j] = *reinterpret_cast<const uint4*>((const T*)a.y + off);
            }
        }
    }
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float amx[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const int n = nin[j];
        if (n <= 0) continue;
        float s0, s1, s3, m;
        reduce_vec<T, NT, RES>(a, ch[j], n, rg[j], rv[j], rr[j], ry[j], s0, s1, s3, m);
        const int seg = rw[j] != row0 ? 1 : 0;
        acc[seg][0] += s0; acc[seg][1] += s1; acc[seg][2] += s0; acc[seg][3] += s3;
        amx[seg] = fmaxf(amx[seg], m);
    }
#pragma unroll
    for (int seg = 0; seg < 2; ++seg) {
        const int r = row0 + seg;
        const uint32_t rfirst = (uint32_t)r * (uint32_t)vpr;           // first vector of row r
        if (seg == 1 && rfirst >= warp_first + 32u * V) break;         // warp lies inside one row (uniform)
        float v[4] = {acc[seg][0], acc[seg][1], RES == 2 ? acc[seg][2] : 0.f, RES == 2 ? acc[seg][3] : 0.f};
#pragma unroll
        for (int i = 0; i < (RES == 2 ? 4 : 2); ++i) v[i] = warp_sum(v[i]);
        const float m = a.gmax ? warp_max(amx[seg]) : 0.f;
        if (lane == 0 && rfirst < tot) {
            const int slot = (int)(wg - rfirst / (32u * V));
            const int b = (int)a.dC.div((uint32_t)r), o = r - b * a.C;
            a.partials[bwd_part_index(a, b, slot, o)] = make_float4(v[0], v[1], v[2], v[3]);
            if (a.gmax) a.amax_part[bwd_part_index(a, b, slot, o)] = m;
        }
    }
}

// ---- channel-per-CTA backward reduction ----------------------------------------------------------------
// One CTA streams channel o of every sample: B * vpr 8-frame vectors, numbered sample-major, thread t the vectors
// t, t + blockDim, ... in batches of U independent 16-byte loads per tensor, sums in registers.  Because the CTA sees
// the whole channel it needs no per-row partials and no finalize launch: it ends with the channel's coefficients.
// (The same mapping was measured for the two apply kernels and lost to the flattened one: a CTA that hops between
// the 32 rows of a channel streams about 10 % slower than one that walks the tensor in address order, and a forward
// apply that merges the contraction's statistics partials in its prologue pays that merge once per CTA.)
constexpr int kChThreads = 512;
// One round of two vectors per thread and one wave of two CTAs per SM (148 of them): with more of either the flattened kernel
// streams faster by more than the launch costs (800 vectors in 512 channels: 94.5 us with two kernels, 95.2 with one).
constexpr int kApplyChVectors = 2 * kChThreads, kApplyChChannels = 2 * 148;

// Merge of the contraction's statistics partials and the apply step, one CTA per channel: one launch instead of two.  A thread
// takes one of the partials (there are at most 320) while its vectors are on their way; the sums are taken in the order of
// bn_finalize_flat_kernel, so the statistics do not depend on which of the two a block takes.  Latency-bound like the chain it
// belongs to.  Blocks forward and backward: 256 channels, 2 x 160 frames 39.9 -> 37.9 us; the same with 8 x 400 57.0 -> 55.4.
template <typename T, typename NT, int RES>
__global__ void __launch_bounds__(kChThreads, 2) bn_apply_ch_kernel(ApplyArgs a, FlatStats f, int vpr) {
    constexpr int NT_ = kChThreads, U = 2;
    __shared__ float2 s_part[kFlatParts * kFinWarps], s_red[kFinWarps];
    const int o = blockIdx.x, tid = threadIdx.x;
    const FlatShare F(f.blk_off[a.B], f.tiles_m, f.G, o / f.rows_per_tile);
    const bool part = F.takes_part(tid);
    const float N = (float)(*f.nvalid);
    FwdChan c{0.f, 0.f, a.gamma[o], a.beta[o], 0.f, 0.f, 0.f, 0.f};
    const int nvec = a.B * vpr;      // at most U * NT_
    int nin[U]; size_t off[U]; uint4 rv[U], rr[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int j = tid + u * NT_;
        nin[u] = -1; off[u] = 0;
        if (j < nvec) {
            const int b = (int)a.dvpr.div((uint32_t)j), t0 = (j - b * vpr) * 8;
            nin[u] = max(0, min(a.len_out[b], a.Tp) - t0);
            off[u] = ((size_t)b * a.C + o) * a.Tp + t0;
        }
    }
    pdl_sync();              // launch_early: lengths, offsets and parameters (read above) were settled before the contraction
    const float4 pv = F.last >= 0 ? f.partials[(size_t)F.first * a.C + o] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 v = part ? f.partials[(size_t)tid * a.C + o] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (nin[u] <= 0) continue;
        rv[u] = *reinterpret_cast<const uint4*>((const NT*)a.v + off[u]);
        if (RES == 1) rr[u] = *reinterpret_cast<const uint4*>((const T*)a.xres + off[u]);
        if (RES == 2) rr[u] = *reinterpret_cast<const uint4*>((const NT*)a.vr + off[u]);
    }
    if (RES == 2) { c.mur = a.mean_r[o]; c.isr = a.invstd_r[o]; c.gar = a.gamma_r[o]; c.ber = a.beta_r[o]; }
    const float pivot = pv.x > 0.f ? pv.y / pv.x : 0.f;
    if (tid < kFlatParts * kFinWarps) {
        const float d = v.x > 0.f ? v.y / v.x - pivot : 0.f;
        s_part[tid] = make_float2(v.x > 0.f ? v.y : 0.f, v.x > 0.f ? fmaf(v.x * d, d, v.z) : 0.f);
    }
    __syncthreads();
    if (tid < kFinWarps) {
        float s1 = 0.f, q = 0.f;
#pragma unroll
        for (int i = 0; i < kFlatParts; ++i) { s1 += s_part[tid + i * kFinWarps].x; q += s_part[tid + i * kFinWarps].y; }
        s_red[tid] = make_float2(s1, q);
    }
    __syncthreads();
    float t = 0.f, m2 = 0.f, var;
#pragma unroll
    for (int i = 0; i < kFinWarps; ++i) { t += s_red[i].x; m2 += s_red[i].y; }
    merged_stats(N, t, m2, pivot, c.mu, var);
    c.is = 1.f / sqrtf(var + f.eps);
    if (tid == 0) put_stats(o, c.mu, c.is, var, N, f.momentum, f.mean, f.invstd, f.running_mean, f.running_var);
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (nin[u] >= 0) apply_core<T, NT, RES>((T*)a.y + off[u], nin[u], rv[u], rr[u], c);
}

// Backward reduction of channel o over every sample, then the channel's coefficients, parameter gradients and its
// term of the bound on |gv| (what bn_bwd_finalize_kernel does for the row-mapped reduction).
template <typename T, typename NT, int RES, int G>
__global__ void __launch_bounds__(kChThreads, G == 2 && RES == 2 ? 1 : 2)
bn_bwd_reduce_ch_kernel(BnBwdArgs a, int vpr, const float* gamma_r, float* dgamma, float* dbeta, float* dgamma_r,
                        float* dbeta_r, int accumulate) {
    constexpr int NT_ = kChThreads;
    // 16-byte loads in flight per thread: U * (2 to 4 tensors) * (1 to 3 vectors)
    constexpr int U = G == 0 ? (RES == 2 ? 2 : 4) : (G == 1 && RES == 0 ? 2 : 1);
    __shared__ float4 s_sum[NT_ / 32];
    const int o = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    BwdChan c{};
    if (RES == 0) { c.ga = a.gamma[o]; c.be = a.beta[o]; }       // the caller's parameters
    pdl_sync();
    // the statistics may come from the kernel just before this one: the last layer's bn_apply_ch_kernel writes them itself
    c.mu = a.mean[o]; c.is = a.invstd[o];
    if (RES == 2) { c.mur = a.mean_r[o]; c.isr = a.invstd_r[o]; }
    const int nvec = a.B * vpr;
    float s0 = 0.f, s1 = 0.f, s3 = 0.f, amax = 0.f;
    for (int jb = tid; jb < nvec; jb += U * NT_) {
        int nin[U];
        BwdRaw<G> rg[U], rv[U], rr[U], ry[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = jb + u * NT_;
            nin[u] = 0;
            if (j < nvec) {
                const int b = (int)a.dvpr.div((uint32_t)j), t0 = (j - b * vpr) * 8;
                nin[u] = max(0, min(a.len_out[b], a.Tp) - t0);
                if (nin[u] > 0) {
                    const size_t off = ((size_t)b * a.C + o) * a.Tp + t0;
                    rg[u] = BwdRaw<G>(a, a.g, off, b, o, t0);
                    rv[u] = BwdRaw<G>(a, a.v, off, b, o, t0);
                    if (RES == 2) rr[u] = BwdRaw<G>(a, a.vr, off, b, o, t0);
                    if (RES != 0) ry[u] = BwdRaw<G>(a, a.y, off, b, o, t0);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (nin[u] <= 0) continue;
            float q0, q1, q3, m;
            reduce_core<T, NT, RES>(nin[u], rg[u].get(nin[u]), rv[u].get(nin[u]), rr[u].get(nin[u]), ry[u].get(nin[u]), c, q0, q1, q3, m);
            s0 += q0; s1 += q1; s3 += q3; amax = fmaxf(amax, m);
        }
    }
    s0 = warp_sum(s0); s1 = warp_sum(s1);
    if (RES == 2) s3 = warp_sum(s3);
    if (a.gmax) amax = warp_max(amax);
    if (lane == 0) s_sum[w] = make_float4(s0, s1, s3, amax);
    __syncthreads();
    if (tid != 0) return;
    float d0 = 0.f, d1 = 0.f, d3 = 0.f;
    amax = 0.f;
#pragma unroll
    for (int i = 0; i < NT_ / 32; ++i) {                // warp order: bit-repeatable
        const float4 q = s_sum[i];
        d0 += q.x; d1 += q.y; d3 += q.z; amax = fmaxf(amax, q.w);
    }
    const float N = (float)(*a.nvalid);
    const float k = a.gamma[o] * c.is;
    const float kr = RES == 2 ? gamma_r[o] * c.isr : 0.f;
    if (a.gmax) {            // see bn_bwd_finalize_kernel
        float bound = fabsf(k) * (amax + fabsf(d0) / N + sqrtf(N) * fabsf(d1) / N);
        if (RES == 2) bound = fmaxf(bound, fabsf(kr) * (amax + fabsf(d0) / N + sqrtf(N) * fabsf(d3) / N));
        if (bound < 3.0e38f) atomicMax(reinterpret_cast<unsigned int*>(a.gmax), __float_as_uint(bound));
    }
    auto put = [&](float* dst, float val) {
        if (dst) dst[o] = accumulate ? dst[o] + val : val;
    };
    put(dbeta, d0); put(dgamma, d1);
    a.coef[o] = make_float4(k, d0 / N, d1 / N, 0.f);
    if (RES == 2) {
        put(dbeta_r, d0); put(dgamma_r, d3);            // the residual sum receives the same gated gradient
        a.coef_r[o] = make_float4(kr, d0 / N, d3 / N, 0.f);
    }
}

template <typename T>
__global__ void __launch_bounds__(kRowThreads)
ew_add_masked_kernel(T* out, const T* a, const T* b, const T* c, const int* len, int nrows, int C, int Tt) {
    pdl_sync();
    SC_ROW_SETUP(nrows)
    const int bb = row / C;
    const int l = min(len[bb], Tt);
    const bool vec = (Tt % 8 == 0);
    const size_t off = (size_t)row * Tt;
    for (int t0 = lane * 8; t0 < Tt; t0 += 256) {
        float f[8];
        if (t0 < l) {
            load_chunk(a + off, t0, Tt, vec, f);
            if (b) { float q[8]; load_chunk(b + off, t0, Tt, vec, q);
#pragma unroll
                for (int i = 0; i < 8; ++i) f[i] += q[i]; }
            if (c) { float q[8]; load_chunk(c + off, t0, Tt, vec, q);
#pragma unroll
                for (int i = 0; i < 8; ++i) f[i] += q[i]; }
#pragma unroll
            for (int i = 0; i < 8; ++i) if (t0 + i >= l) f[i] = 0.f;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) f[i] = 0.f;
        }
        store_chunk(out + off, t0, Tt, vec, f);
    }
}

}  // namespace

#define SC_DISPATCH3(dtype, ...)                                                              \
    switch (dtype) {                                                                          \
        case F32: { using T = float; using NT = float; __VA_ARGS__; break; }                  \
        case F16: { using T = __half; using NT = __half; __VA_ARGS__; break; }                \
        default:  { using T = __nv_bfloat16; using NT = __half; __VA_ARGS__; break; }         \
    }
// 16-bit activation types only (the flattened kernels move 16-byte vectors of 8 elements)
#define SC_DISPATCH16(dtype, ...)                                                             \
    if (dtype == F16) { using T = __half; using NT = __half; __VA_ARGS__; }                   \
    else { using T = __nv_bfloat16; using NT = __half; __VA_ARGS__; }
#define SC_DISPATCH(dtype, ...)                                             \
    switch (dtype) {                                                        \
        case F32: { using T = float; __VA_ARGS__; break; }                  \
        case F16: { using T = __half; __VA_ARGS__; break; }                 \
        default:  { using T = __nv_bfloat16; __VA_ARGS__; break; }          \
    }

void prologue(const Launch& L, Prologue& p) {
    double bytes = 8.0 * p.B * p.phases;
    int blocks = 0;
    for (int k = 0; k < p.conv.count; ++k) {
        p.conv.first[k] = blocks;
        blocks += (p.conv.n[k] + kConvertChunk - 1) / kConvertChunk; bytes += 4.0 * p.conv.n[k];
    }
    KScope ks_(L, KC_LENGTHS, bytes, 0.0);
    launch_k(L, prologue_kernel, 1 + blocks, kLenThreads, 0, p, L.status);
    if (L.fresh) L.fresh[L.lane] = true;
    L.count();
}

void bn_stats(const Launch& L, int vdtype, const void* v, const int* len_out, int B, int C, int Tp,
              float2* partials) {
    KScope ks_(L, KC_BN_STATS, (double)dtype_size(vdtype) * B * C * Tp, 0.0);
    if (vdtype == F32) launch_k(L, bn_stats_kernel<float>, (B * C + kRowsPerCta - 1) / kRowsPerCta, kRowThreads, 0, (const float*)v, len_out, B * C, C, Tp, partials);
    else launch_k(L, bn_stats_kernel<__half>, (B * C + kRowsPerCta - 1) / kRowsPerCta, kRowThreads, 0, (const __half*)v, len_out, B * C, C, Tp, partials);
    L.count();
}

void bn_finalize(const Launch& L, const float2* partials, int parts_per_b, int tile_w, const int* len_out,
                 const int* nvalid, int B, int C, float eps, float momentum, float* mean, float* invstd,
                 float* running_mean, float* running_var) {
    KScope ks_(L, KC_BN_FINALIZE, 8.0 * B * parts_per_b * C, 0.0);
    launch_k(L, bn_finalize_kernel, (C + 31) / 32, 32 * kFinWarps, 0, partials, parts_per_b, tile_w, len_out, nvalid, B, C,
                                                                     eps, momentum, mean, invstd, running_mean, running_var);
    L.count();
}

void bn_finalize_flat(const Launch& L, const float4* partials, int grid, int tiles_m, int rows_per_tile,
                      const int* blk_off, const int* nvalid, int B, int C, float eps, float momentum, float* mean,
                      float* invstd, float* running_mean, float* running_var) {
    KScope ks_(L, KC_BN_FINALIZE, 16.0 * grid * C / std::max(1, tiles_m), 0.0);
    launch_early(L, bn_finalize_flat_kernel, (C + 31) / 32, 32 * kFinWarps, 0, partials, grid, tiles_m, rows_per_tile, blk_off, nvalid, B,
                                                                          C, eps, momentum, mean, invstd, running_mean, running_var);
    L.count();
}

bool bn_small(int dtype, int B, int C, int Tp) {
    const long long chunks = (long long)B * ((Tp + 7) / 8);
    return dtype == F32 && chunks <= kSmallChunks &&
           (Tp % 8 == 0 || B <= kSmallOddSamples || (chunks <= kSmallOddChunks && chunks * C <= kSmallOddWork));
}

void bn_small_fwd(const Launch& L, const ApplyArgs& a, const int* nvalid, float eps, float momentum, float* mean, float* invstd,
                  float* running_mean, float* running_var) {
    KScope ks_(L, KC_BN_APPLY, 4.0 * a.B * a.C * a.Tp * (a.residual ? 3 : 2), 0.0);
    launch_early(L, bn_small_fwd_kernel, (unsigned)a.C, kRowThreads, 0, a, nvalid, eps, momentum, mean, invstd, running_mean, running_var);
    L.count();
}

// the flattened kernels index with 32 bits
static bool fits32(int B, int C, int Tp) { return (long long)B * C * (Tp / 8) < (1ll << 31) && (long long)B * C * Tp < (1ll << 31); }
static unsigned fast_grid(long long total, int V) { return (unsigned)((total + 256ll * V - 1) / (256ll * V)); }

// Algorithmic bytes per element of the batch-norm kernels: every tensor they must read or write, once.
// The channel-per-CTA reduction: one launch instead of two, which wins unless the tensor is large and its channels are too few
// for their CTAs (two per SM) to stream as fast as the flattened kernel does on all SMs.  Blocks forward and backward without a
// depthwise step, bf16: time with the flattened kernel and its finalize step over time with this one,
//   at any width up to 4096 vectors per channel                          1.00-1.08 (identity residual, rows of 1600: 0.97-1.03)
//   rows of 2048 frames and more: 8 to 24 channels, 8192 / 32768 vectors 0.96-0.98 / 0.90-0.94
//                                 32 channels                            0.99 / 0.95      (identity, 8192: 0.92)
//                                 64 channels                            1.01 / 0.99      (identity, 8192: 0.94)
//                                 96 channels and more                   1.03-1.09        (identity, rows of 1600: 0.97-1.02)
//   16 to 48 channels, 8192 and 16384 vectors: rows of 512 frames        1.04-1.09
//                                              rows of 1024              0.98-1.04
//   rows of 128 and 256 frames, 2048 to 16384 vectors                    0.97-1.21, below 1 only in 8 channels of 128 frames
static bool channel_mapped(int B, int C, int Tp) { return C >= 64 || Tp < 2048 || (long long)B * (Tp / 8) <= 4096; }
static_assert(2048 / 8 >= kRedVectors, "a warp of the flattened reduction meets at most two rows");

void bn_apply(const Launch& L, int dtype, const ApplyArgs& a_in) {
    ApplyArgs a = a_in;
    const double e = (double)dtype_size(dtype), en = (double)dtype_size(ntype_of(dtype));
    KScope ks_(L, KC_BN_APPLY, (double)a.B * a.C * (a.phases ? a.T : a.Tp) * (en + e + (a.residual == 1 ? e : 0) + (a.residual == 2 ? en : 0)), 0.0);
    if (a.phases) {
        a.dT = FastDiv((uint32_t)a.T);
        const uint32_t total = (uint32_t)a.B * a.C * a.T, total_u = a.u_out ? (uint32_t)a.B * a.Cu * a.T : 0;
        const int nba = (int)fast_grid((total + 7) / 8, 1);
        const unsigned grid = nba + (a.u_out ? fast_grid((total_u + 7) / 8, 1) : 0);
#define SC_APPLY_UNPACK(RES)                                                                                                  \
        if (a.phases == 2) { SC_DISPATCH16(dtype, (launch_early(L, bn_apply_unpack_kernel<T, NT, RES, 2>, grid, 256, 0, a, total, nba, total_u))) } \
        else { SC_DISPATCH16(dtype, (launch_early(L, bn_apply_unpack_kernel<T, NT, RES, 1>, grid, 256, 0, a, total, nba, total_u))) }
        if (a.residual == 0) { SC_APPLY_UNPACK(0) } else if (a.residual == 1) { SC_APPLY_UNPACK(1) } else { SC_APPLY_UNPACK(2) }
#undef SC_APPLY_UNPACK
        L.count();
        return;
    }
    if (dtype != F32 && a.Tp % 8 == 0 && a.has_relu && a.res_before_relu && fits32(a.B, a.C, a.Tp)) {
        const int vpr = a.Tp / 8;
        a.dvpr = FastDiv((uint32_t)vpr); a.dC = FastDiv((uint32_t)a.C);
        const long long total = (long long)a.B * a.C * vpr;
        const unsigned grid = fast_grid(total, 2);
#define SC_APPLY_FAST(RES) SC_DISPATCH16(dtype, (launch_early(L, bn_apply_fast_kernel<T, NT, RES, 2>, grid, 256, 0, a, vpr, total)))
        if (a.residual == 0) { SC_APPLY_FAST(0); } else if (a.residual == 1) { SC_APPLY_FAST(1); } else { SC_APPLY_FAST(2); }
#undef SC_APPLY_FAST
        L.count();
        return;
    }
    SC_DISPATCH3(dtype, (launch_k(L, bn_apply_kernel<T, NT>, (a.B * a.C + kRowsPerCta - 1) / kRowsPerCta, kRowThreads, 0, a)));
    L.count();
}

bool bn_apply_takes_stats(int dtype, const ApplyArgs& a) {
    return dtype != F32 && !a.phases && a.Tp % 8 == 0 && a.has_relu && a.res_before_relu && fits32(a.B, a.C, a.Tp) &&
           (long long)a.B * (a.Tp / 8) <= kApplyChVectors && a.C <= kApplyChChannels;
}
void bn_apply_flat(const Launch& L, int dtype, const ApplyArgs& a_in, const FlatStats& f) {
    ApplyArgs a = a_in;
    const double e = (double)dtype_size(dtype), en = (double)dtype_size(ntype_of(dtype));
    KScope ks_(L, KC_BN_APPLY, (double)a.B * a.C * a.Tp * (en + e + (a.residual == 1 ? e : 0) + (a.residual == 2 ? en : 0)), 0.0);
    const int vpr = a.Tp / 8;
    a.dvpr = FastDiv((uint32_t)vpr);
    if (a.residual == 0) { SC_DISPATCH16(dtype, (launch_early(L, bn_apply_ch_kernel<T, NT, 0>, (unsigned)a.C, kChThreads, 0, a, f, vpr))); }
    else if (a.residual == 1) { SC_DISPATCH16(dtype, (launch_early(L, bn_apply_ch_kernel<T, NT, 1>, (unsigned)a.C, kChThreads, 0, a, f, vpr))); }
    else { SC_DISPATCH16(dtype, (launch_early(L, bn_apply_ch_kernel<T, NT, 2>, (unsigned)a.C, kChThreads, 0, a, f, vpr))); }
    L.count();
}

static void bn_bwd_reduce(const Launch& L, int dtype, BnBwdArgs& a) {
    a.nslots = 1;
    const double e = (double)dtype_size(dtype), en = (double)dtype_size(ntype_of(dtype));
    if (dtype != F32 && a.Tp % 8 == 0 && a.has_bn && a.has_relu && a.res_before_relu && fits32(a.B, a.C, a.Tp)) {
        a.dvpr = FastDiv((uint32_t)(a.Tp / 8)); a.dC = FastDiv((uint32_t)a.C);
        KScope ks2_(L, KC_BN_BWD_REDUCE, (double)a.B * a.C * a.Tp * (e * (a.residual == 0 ? 1 : 2) + en * (a.residual == 2 ? 2 : 1)), 0.0);
        const int vpr = a.Tp / 8;
        a.nslots = bn_bwd_max_slots(a.Tp);
        const long long total = (long long)a.B * a.C * vpr;
        const unsigned grid = fast_grid(total, kRedV);
#define SC_RED_FAST(RES) SC_DISPATCH16(dtype, (launch_k(L, bn_bwd_reduce_fast_kernel<T, NT, RES>, grid, 256, 0, a, vpr, total)))
        if (a.residual == 2) { SC_RED_FAST(2); } else if (a.residual == 1) { SC_RED_FAST(1); } else { SC_RED_FAST(0); }
#undef SC_RED_FAST
        L.count();
        return;
    }
    KScope ks_(L, KC_BN_BWD_REDUCE, (double)a.B * a.C * a.Tp * (e * (a.has_relu && a.res_before_relu ? 2 : 1) + (a.has_bn ? en : 0) + (a.residual == 2 ? en : 0)), 0.0);
    SC_DISPATCH3(dtype, (launch_k(L, bn_bwd_reduce_kernel<T, NT>, (a.B * a.C + kRowsPerCta - 1) / kRowsPerCta, kRowThreads, 0, a)));
    L.count();
}

static void bn_bwd_finalize(const Launch& L, const BnBwdArgs& a, const float* gamma, const float* gamma_r,
                     float* dgamma, float* dbeta, float* dgamma_r, float* dbeta_r, float* dbias,
                     int accumulate) {
    KScope ks_(L, KC_BN_BWD_FINALIZE, 16.0 * a.B * a.C * a.nslots, 0.0);
    launch_k(L, bn_bwd_finalize_kernel, (a.C + 31) / 32, 32 * kFinWarps, 0, a, BwdGrads{gamma, gamma_r, dgamma, dbeta, dgamma_r, dbeta_r, dbias, accumulate});
    L.count();
}

static void bn_bwd_reduce_finalize(const Launch& L, int dtype, BnBwdArgs& a, const float* gamma, const float* gamma_r,
                            float* dgamma, float* dbeta, float* dgamma_r, float* dbeta_r, float* dbias, int accumulate) {
    const bool fast = dtype != F32 && a.Tp % 8 == 0 && a.has_bn && a.has_relu && a.res_before_relu && fits32(a.B, a.C, a.Tp);
    if (a.phases || (fast && channel_mapped(a.B, a.C, a.Tp))) {
        a.nslots = 1;
        const double e = (double)dtype_size(dtype), en = (double)dtype_size(ntype_of(dtype));
        KScope ks_(L, KC_BN_BWD_REDUCE, (double)a.B * a.C * a.Tp * (e * (a.residual == 0 ? 1 : 2) + en * (a.residual == 2 ? 2 : 1)), 0.0);
        const int vpr = a.Tp / 8;
        a.dvpr = FastDiv((uint32_t)vpr);
#define SC_RED_CH_G(RES, G) SC_DISPATCH16(dtype, (launch_k(L, bn_bwd_reduce_ch_kernel<T, NT, RES, G>, (unsigned)a.C, kChThreads, 0, a, vpr, \
                                                          gamma_r, dgamma, dbeta, dgamma_r, dbeta_r, accumulate)))
#define SC_RED_CH(RES) if (a.phases == 2) { SC_RED_CH_G(RES, 2) } else if (a.phases == 1) { SC_RED_CH_G(RES, 1) } else { SC_RED_CH_G(RES, 0) }
        if (a.residual == 2) { SC_RED_CH(2) } else if (a.residual == 1) { SC_RED_CH(1) } else { SC_RED_CH(0) }
#undef SC_RED_CH_G
#undef SC_RED_CH
        L.count();
        return;
    }
    bn_bwd_reduce(L, dtype, a);
    bn_bwd_finalize(L, a, gamma, gamma_r, dgamma, dbeta, dgamma_r, dbeta_r, dbias, accumulate);
}

static void bn_bwd_apply(const Launch& L, int dtype, const BnBwdArgs& a_in) {
    BnBwdArgs a = a_in;
    const bool fast_apply = dtype != F32 && a.Tp % 8 == 0 && a.has_bn && a.has_relu && a.res_before_relu && fits32(a.B, a.C, a.Tp);
    const double e = (double)dtype_size(dtype), en = (double)dtype_size(ntype_of(dtype));
    KScope ks_(L, KC_BN_BWD_APPLY, (double)a.B * a.C * a.Tp * (e * (a.has_relu && a.res_before_relu && !(fast_apply && a.residual == 0) ? 2 : 1) + (a.has_bn ? en : 0) + (a.residual == 2 ? en : 0) + (double)dtype_size(a.gv_dtype) + (a.residual != 0 ? e : 0)), 0.0);
    if (fast_apply) {
        const int vpr = a.Tp / 8;
        a.dvpr = FastDiv((uint32_t)vpr); a.dC = FastDiv((uint32_t)a.C);
        const long long total = (long long)a.B * a.C * vpr;
        const unsigned grid = fast_grid(total, a.phases ? 1 : 2);
#define SC_BWD_FAST_G(RES, G)                                                                                        \
        if (dtype == BF16 && a.gv_dtype == F16)                                                                      \
            launch_early(L, bn_bwd_apply_fast_kernel<__nv_bfloat16, __half, __half, RES, (G ? 1 : 2), G>, grid, 256, 0, a, vpr, total); \
        else { SC_DISPATCH16(dtype, (launch_early(L, bn_bwd_apply_fast_kernel<T, NT, T, RES, (G ? 1 : 2), G>, grid, 256, 0, a, vpr, total))); }
#define SC_BWD_FAST(RES) if (a.phases == 2) { SC_BWD_FAST_G(RES, 2) } else if (a.phases == 1) { SC_BWD_FAST_G(RES, 1) } else { SC_BWD_FAST_G(RES, 0) }
        if (a.residual == 0) { SC_BWD_FAST(0) } else if (a.residual == 1) { SC_BWD_FAST(1) } else { SC_BWD_FAST(2) }
#undef SC_BWD_FAST
#undef SC_BWD_FAST_G
        L.count();
        return;
    }
    if (dtype == BF16 && a.gv_dtype == F16)
        launch_k(L, bn_bwd_apply_kernel<__nv_bfloat16, __half, __half>, (a.B * a.C + kRowsPerCta - 1) / kRowsPerCta, kRowThreads, 0, a);
    else
        SC_DISPATCH3(dtype, (launch_k(L, bn_bwd_apply_kernel<T, NT, T>, (a.B * a.C + kRowsPerCta - 1) / kRowsPerCta, kRowThreads, 0, a)));
    L.count();
}

void bn_bwd(const Launch& L, int dtype, BnBwdArgs& a, const float* gamma, const float* gamma_r, float* dgamma, float* dbeta,
            float* dgamma_r, float* dbeta_r, float* dbias, int accumulate) {
    if (bn_small(dtype, a.B, a.C, a.Tp)) {
        KScope ks_(L, KC_BN_BWD_APPLY, 4.0 * a.B * a.C * a.Tp * (a.residual ? 5 : 4), 0.0);
        launch_k(L, bn_small_bwd_kernel, (unsigned)a.C, kRowThreads, 0, a, BwdGrads{gamma, gamma_r, dgamma, dbeta, dgamma_r, dbeta_r, dbias, accumulate});
        L.count();
        return;
    }
    bn_bwd_reduce_finalize(L, dtype, a, gamma, gamma_r, dgamma, dbeta, dgamma_r, dbeta_r, dbias, accumulate);
    bn_bwd_apply(L, dtype, a);
}

void ew_add_masked(const Launch& L, int dtype, void* out, const void* a, const void* b, const void* c,
                   const int* len, int B, int C, int Tt) {
    KScope ks_(L, KC_EW, (double)dtype_size(dtype) * B * C * Tt * (2 + (b ? 1 : 0) + (c ? 1 : 0)), 0.0);
    SC_DISPATCH(dtype, (launch_k(L, ew_add_masked_kernel<T>, (B * C + kRowsPerCta - 1) / kRowsPerCta, kRowThreads, 0, (T*)out, (const T*)a, (const T*)b,
                                                                                      (const T*)c, len, B * C, C, Tt)));
    L.count();
}

namespace {
// one 8-frame vector per thread (rows are a multiple of 8 frames) or one element per thread
__global__ void __launch_bounds__(256)
mask_convert_f16_kernel(__half* __restrict__ out, const __nv_bfloat16* __restrict__ in, const int* __restrict__ len,
                        int C, int Tt, long long total, int vec, int* status) {
    pdl_sync();
    const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
    if (idx >= total) return;
    const int per_row = vec ? Tt / 8 : Tt;
    const long long row = idx / per_row;
    const int t0 = (int)(idx - row * per_row) * (vec ? 8 : 1);
    const int l = min(len[row / C], Tt);
    const size_t off = (size_t)row * Tt + t0;
    bool over = false;
    if (vec) {
        float f[8];
        if (t0 < l) {
            ld8<__nv_bfloat16>(in + off, f);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (t0 + i >= l) f[i] = 0.f;
                if (fabsf(f[i]) > 65504.f) { f[i] = copysignf(65504.f, f[i]); over = true; }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) f[i] = 0.f;
        }
        st8<__half>(out + off, f);
    } else {
        float f = t0 < l ? __bfloat162float(in[off]) : 0.f;
        if (fabsf(f) > 65504.f) { f = copysignf(65504.f, f); over = true; }
        out[off] = __float2half_rn(f);
    }
    if (over) raise_status(status, kErrRange);
}
}  // namespace

void mask_convert_f16(const Launch& L, void* out, const void* in, const int* len, int B, int C, int Tt) {
    KScope ks_(L, KC_EW, 4.0 * B * C * Tt, 0.0);
    const int vec = (Tt % 8 == 0) ? 1 : 0;
    const long long total = (long long)B * C * (vec ? Tt / 8 : Tt);
    launch_k(L, mask_convert_f16_kernel, (unsigned)((total + 255) / 256), 256, 0, (__half*)out, (const __nv_bfloat16*)in, len,
                                                                                C, Tt, total, vec, L.status);
    L.count();
}

void mask_copy(const Launch& L, int dtype, void* out, const void* in, const int* len, int B, int C, int Tt) {
    ew_add_masked(L, dtype, out, in, nullptr, nullptr, len, B, C, Tt);
}

}  // namespace sc
