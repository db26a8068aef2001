// Operand copies around the tensor-core form of the non-separable convolution (tc_gemm.cu, CONV modes): activations to
// time-major [B, T, C], weights [C_out, C_in, K] to one matrix per tap, and the sum of the weight gradient's slices back to
// [C_out, C_in, K].  All are pure data movement through L2: the tensors of one call are a few megabytes.
// The whole block, 16 samples x 400 frames, 256 -> 256, K = 11, fp16, forward + backward: 1710 us with the SIMT
// convolution (10 TFLOP/s), 115 us now: the three contractions take 22 + 21 + 17 us (400-540 TFLOP/s; every CTA streams the
// whole weight from L2), these copies 26.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace sc {
namespace {

// 64 channels x 64 frames per CTA through shared memory: 16-byte accesses on both sides.  The shared rows are frames; a
// row pitch of 72 elements keeps 16-byte alignment, and channel pairs are written as 32-bit words.
constexpr int kTile = 64, kPitch = 72;
__global__ void __launch_bounds__(256)
time_major_kernel(const unsigned short* __restrict__ in, unsigned short* __restrict__ out, const int* __restrict__ len, int C, int T) {
    pdl_sync();
    __shared__ __align__(16) unsigned short s[kTile][kPitch];
    const int t0 = blockIdx.x * kTile, c0 = blockIdx.y * kTile, b = blockIdx.z, tid = threadIdx.x;
    const int n = min(len[b], T);
    {   // thread: channel pair 2 (tid / 8), frames 8 (tid % 8) .. + 7
        const int c = c0 + 2 * (tid >> 3), t = t0 + 8 * (tid & 7);
        uint4 v[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            v[i] = make_uint4(0, 0, 0, 0);
            if (c + i < C && t < n) {
                v[i] = *reinterpret_cast<const uint4*>(in + ((size_t)b * C + c + i) * T + t);
                if (t + 8 > n) v[i] = keep_first(v[i], n - t);
            }
        }
        const uint32_t a[4] = {v[0].x, v[0].y, v[0].z, v[0].w}, h[4] = {v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 8 * (tid & 7) + 2 * i, k = 2 * (tid >> 3);
            *reinterpret_cast<uint32_t*>(&s[r][k]) = __byte_perm(a[i], h[i], 0x5410);
            *reinterpret_cast<uint32_t*>(&s[r + 1][k]) = __byte_perm(a[i], h[i], 0x7632);
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int r = (tid >> 3) + 32 * i, c = 8 * (tid & 7);
        if (t0 + r < T && c0 + c < C)       // C is a multiple of 8
            *reinterpret_cast<uint4*>(out + ((size_t)b * T + t0 + r) * C + c0 + c) = *reinterpret_cast<const uint4*>(&s[r][c]);
    }
}

// [C_out, C_in, K] -> [K][C_out][C_in] (swap = 0) or [K][C_in][C_out] (swap = 1); the written index runs with the thread
__global__ void __launch_bounds__(256)
taps_kernel(const unsigned short* __restrict__ w, unsigned short* __restrict__ out, int Cout, int Cin, int K, int swap) {
    pdl_sync();
    const int i = blockIdx.x * 256 + threadIdx.x, n = Cout * Cin;
    if (i >= n) return;
    const int o = swap ? i % Cout : i / Cin, c = swap ? i / Cout : i % Cin;
    const unsigned short* p = w + ((size_t)o * Cin + c) * K;
    for (int k = 0; k < K; ++k) out[(size_t)k * n + i] = p[k];
}

// out[i][k] (+)= sum_s part[s][k][i], in slice order.  A CTA takes 32 rows i (one per lane, so the reads of a warp are one
// 128-byte line) with its eight warps on different taps, and writes the rows as one run through shared memory.  (256 rows
// per CTA with a thread per row: 37 us where this takes 8, too few loads in flight.)
__global__ void __launch_bounds__(256)
reduce_taps_kernel(const float* __restrict__ part, int nsplit, int n, int K, int kchunk, float* __restrict__ out, int accumulate) {
    pdl_sync();
    extern __shared__ float s[];              // [32][kchunk]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, i = i0 + lane, rows = min(32, n - i0);
    for (int k0 = 0; k0 < K; k0 += kchunk) {
        const int kn = min(kchunk, K - k0);
        if (i < n) {
            for (int k = w; k < kn; k += 8) {
                const float* p = part + (size_t)(k0 + k) * n + i;
                float v = 0.f;
                int q = 0;
                for (; q + 4 <= nsplit; q += 4) {
                    float x[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) x[e] = p[(size_t)(q + e) * K * n];
#pragma unroll
                    for (int e = 0; e < 4; ++e) v += x[e];
                }
                for (; q < nsplit; ++q) v += p[(size_t)q * K * n];
                s[lane * kn + k] = v;
            }
        }
        __syncthreads();
        for (int e = threadIdx.x; e < rows * kn; e += 256) {
            const size_t at = (size_t)(i0 + e / kn) * K + k0 + e % kn;
            out[at] = accumulate ? out[at] + s[e] : s[e];
        }
        __syncthreads();
    }
}

}  // namespace

void to_time_major(const Launch& L, const void* in, void* out, const int* len, int B, int C, int T) {
    KScope ks_(L, KC_EW, 4.0 * B * C * T, 0.0);
    launch_k(L, time_major_kernel, dim3((T + kTile - 1) / kTile, (C + kTile - 1) / kTile, B), 256, 0, (const unsigned short*)in,
             (unsigned short*)out, len, C, T);
    L.count();
}

void split_taps(const Launch& L, const void* w, void* out, int Cout, int Cin, int K, int swap) {
    KScope ks_(L, KC_EW, 4.0 * Cout * Cin * K, 0.0);
    launch_k(L, taps_kernel, (unsigned)(((long long)Cout * Cin + 255) / 256), 256, 0, (const unsigned short*)w, (unsigned short*)out, Cout,
             Cin, K, swap);
    L.count();
}

void conv_reduce_taps(const Launch& L, const float* partials, int nsplit, int n, int K, float* out, int accumulate) {
    KScope ks_(L, KC_REDUCE, 4.0 * (nsplit + 1) * (double)n * K, 0.0);
    const int kchunk = std::min(K, 32);
    launch_k(L, reduce_taps_kernel, (unsigned)((n + 31) / 32), 256, (size_t)32 * kchunk * sizeof(float), partials, nsplit, n, K, kchunk,
             out, accumulate);
    L.count();
}

}  // namespace sc
