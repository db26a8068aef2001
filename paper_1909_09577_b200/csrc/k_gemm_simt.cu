// Pointwise (1x1) convolution as plain SIMT tiled GEMMs with fp32 accumulation.
// These serve the fp32 path (whose tolerance rules out reduced-precision tensor-core formats) and
// any shape the tensor-core kernels do not tile.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace sc {
namespace {

// D[m,n] = sum_k A(m,k) * B(k,n) for one z-slice; operand access is described by strides so that the
// three contractions (forward, input gradient, weight gradient) share the kernel.
struct GemmDesc {
    int M, N, Kd;
    // A(m,k) = a[z*a_z + m*a_m + k*a_k];  B(k,n) = b[z*b_z + k*b_k + n*b_n]
    long long a_z, a_m, a_k, b_z, b_k, b_n;
    int per_z, k_len;                 // weight gradient: slice z = sample * per_z + i covers the frames [i k_len, (i+1) k_len) of the sample
};

template <typename X> struct IsHalf { static constexpr bool value = false; };
template <> struct IsHalf<__half> { static constexpr bool value = true; };

constexpr int BK = 32, NT = 256;

// TS x TS output tile (64: 4 x 4 per thread; 32: 2 x 2, for problems of few tiles).  The next 32-deep step travels through
// registers while the current one is computed (two shared-memory buffers, one barrier per step): with the loads between two
// barriers a step cost two round trips to L2 (64 x 64 x 128 frames, two samples, fp32: forward 11.3 -> 3.4 us, input gradient
// 11.0 -> 2.9, weight gradient 24.8 -> 2.4, the last one also with several slices per sample).  Every output sums k in increasing order.
// MODE 0: fwd (bias+mask, OT out) 1: dgrad (OT out) 2: wgrad (float partial out)
template <typename T, typename OT, int MODE, int TS>
__global__ void __launch_bounds__(NT)
gemm_simt_kernel(GemmDesc d, const T* __restrict__ a, const T* __restrict__ b, void* __restrict__ out,
                 const float* __restrict__ bias, const int* __restrict__ len_out, int* status) {
    constexpr int R = TS / 16, PER = TS * BK / NT;
    __shared__ __align__(16) float As[2][BK][TS + 4];
    __shared__ __align__(16) float Bs[2][BK][TS + 4];
    const int z = blockIdx.z;
    const int m0 = blockIdx.y * TS, n0 = blockIdx.x * TS;
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    float acc[R][R] = {};
    pdl_sync();

    int ke = d.Kd, kb = 0;
    const T* ap = a; const T* bp = b;
    if (MODE == 2) {
        const int zb = z / d.per_z;
        kb = (z - zb * d.per_z) * d.k_len; ke = min(d.Kd, kb + d.k_len);
        ap += (long long)zb * d.a_z; bp += (long long)zb * d.b_z;
    } else {
        ap += (long long)z * d.a_z; bp += (long long)z * d.b_z;
    }

    // fwd-mode early exit: tile wholly in padding -> zeros
    if (MODE == 0 && len_out && n0 >= len_out[z]) {
        OT* o = (OT*)out + (long long)z * d.M * d.N;
        for (int i = tid; i < TS * TS; i += NT) {
            const int m = m0 + i / TS, n = n0 + i % TS;
            if (m < d.M && n < d.N) stf(o + (long long)m * d.N + n, 0.f);
        }
        return;
    }

    // the thread -> element map follows the index that is contiguous in memory
    constexpr bool AK = MODE != 1, BKc = MODE == 2;       // contiguous along k: forward weights, both weight-gradient operands
    float ra[PER], rb[PER];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const int i = tid + e * NT;
            const int am = AK ? i / BK : i % TS, ak = AK ? i % BK : i / TS;
            const int bn = BKc ? i / BK : i % TS, bk = BKc ? i % BK : i / TS;
            ra[e] = (m0 + am < d.M && k0 + ak < ke) ? ldf(ap + (long long)(m0 + am) * d.a_m + (long long)(k0 + ak) * d.a_k) : 0.f;
            rb[e] = (n0 + bn < d.N && k0 + bk < ke) ? ldf(bp + (long long)(k0 + bk) * d.b_k + (long long)(n0 + bn) * d.b_n) : 0.f;
        }
    };
    auto park = [&](int q) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const int i = tid + e * NT;
            As[q][AK ? i % BK : i / TS][AK ? i / BK : i % TS] = ra[e];
            Bs[q][BKc ? i % BK : i / TS][BKc ? i / BK : i % TS] = rb[e];
        }
    };
    fetch(kb);
    park(0);
    __syncthreads();
    int q = 0;
    for (int k0 = kb; k0 < ke; k0 += BK, q ^= 1) {
        const bool more = k0 + BK < ke;
        if (more) fetch(k0 + BK);
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            float aa[R], bb[R];
            if (R == 4) {
                const float4 av = *reinterpret_cast<const float4*>(&As[q][k][ty * 4]), bv = *reinterpret_cast<const float4*>(&Bs[q][k][tx * 4]);
                aa[0] = av.x; aa[1] = av.y; aa[R - 2] = av.z; aa[R - 1] = av.w;
                bb[0] = bv.x; bb[1] = bv.y; bb[R - 2] = bv.z; bb[R - 1] = bv.w;
            } else {
                const float2 av = *reinterpret_cast<const float2*>(&As[q][k][ty * 2]), bv = *reinterpret_cast<const float2*>(&Bs[q][k][tx * 2]);
                aa[0] = av.x; aa[1] = av.y; bb[0] = bv.x; bb[1] = bv.y;
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) acc[i][j] = fmaf(aa[i], bb[j], acc[i][j]);
        }
        if (more) { park(q ^ 1); __syncthreads(); }
    }

#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int m = m0 + ty * R + i;
        if (m >= d.M) continue;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int n = n0 + tx * R + j;
            if (n >= d.N) continue;
            if (MODE == 0) {
                float v = acc[i][j] + (bias ? bias[m] : 0.f);
                if (len_out && n >= len_out[z]) v = 0.f;
                if (sizeof(OT) == 2 && fabsf(v) > 65504.f && IsHalf<OT>::value) { v = copysignf(65504.f, v); raise_status(status, kErrRange); }
                stf((OT*)out + ((long long)z * d.M + m) * d.N + n, v);
            } else if (MODE == 1) {
                stf((OT*)out + ((long long)z * d.M + m) * d.N + n, acc[i][j]);
            } else {
                ((float*)out)[((long long)z * d.M + m) * d.N + n] = acc[i][j];
            }
        }
    }
}

// 64 x 64 tiles where they fill the SMs, else 32 x 32
template <typename T, typename OT, int MODE>
void launch_gemm(const Launch& L, const GemmDesc& d, int nz, const void* a, const void* b, void* out, const float* bias, const int* len) {
    auto tiles = [&](int ts) { return (long long)((d.N + ts - 1) / ts) * ((d.M + ts - 1) / ts) * nz; };
    auto grid = [&](int ts) { return dim3((d.N + ts - 1) / ts, (d.M + ts - 1) / ts, nz); };
    if (tiles(64) >= 148) launch_k(L, gemm_simt_kernel<T, OT, MODE, 64>, grid(64), NT, 0, d, (const T*)a, (const T*)b, out, bias, len, L.status);
    else launch_k(L, gemm_simt_kernel<T, OT, MODE, 32>, grid(32), NT, 0, d, (const T*)a, (const T*)b, out, bias, len, L.status);
}

__global__ void reduce_partials_kernel(const float* __restrict__ p, int nsplit, long long n,
                                       float* __restrict__ out, int accumulate, const float* __restrict__ gmax) {
    pdl_sync();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float s = 0.f;
    for (int k = 0; k < nsplit; ++k) s += p[(long long)k * n + i];
    if (gmax) s *= 1.f / pow2_scale(*gmax);
    out[i] = accumulate ? out[i] + s : s;
}

// Four consecutive elements per thread, eight splits in flight at a time; the order of the additions
// is the same as in the scalar kernel (split 0 first), so both give the same bits.
__global__ void __launch_bounds__(256)
reduce_partials_vec4_kernel(const float4* __restrict__ p, int nsplit, long long n4, float4* __restrict__ out,
                            int accumulate, const float* __restrict__ gmax) {
    pdl_sync();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4) return;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    int k = 0;
    for (; k + 8 <= nsplit; k += 8) {
        float4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = p[(long long)(k + j) * n4 + i];
#pragma unroll
        for (int j = 0; j < 8; ++j) { s.x += v[j].x; s.y += v[j].y; s.z += v[j].z; s.w += v[j].w; }
    }
    for (; k < nsplit; ++k) {
        const float4 v = p[(long long)k * n4 + i];
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    if (gmax) { const float r = 1.f / pow2_scale(*gmax); s.x *= r; s.y *= r; s.z *= r; s.w *= r; }
    if (accumulate) { const float4 o = out[i]; s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w; }
    out[i] = s;
}

}  // namespace

#define SC_DISPATCH(dtype, ...)                                             \
    switch (dtype) {                                                        \
        case F32: { using T = float; __VA_ARGS__; break; }                  \
        case F16: { using T = __half; __VA_ARGS__; break; }                 \
        default:  { using T = __nv_bfloat16; __VA_ARGS__; break; }          \
    }

void reduce_partials(const Launch& L, const float* partials, int nsplit, int64_t n, float* out, int accumulate,
                     const float* gmax) {
    KScope ks_(L, KC_REDUCE, 4.0 * (nsplit + 1) * n, 0.0);
    if (n % 4 == 0 && (reinterpret_cast<uintptr_t>(partials) & 15) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0)
        launch_k(L, reduce_partials_vec4_kernel, (unsigned)((n / 4 + 255) / 256), 256, 0, 
            reinterpret_cast<const float4*>(partials), nsplit, n / 4, reinterpret_cast<float4*>(out), accumulate, gmax);
    else
        launch_k(L, reduce_partials_kernel, (unsigned)((n + 255) / 256), 256, 0, partials, nsplit, n, out, accumulate, gmax);
    L.count();
}

void gemm_fwd_simt(const Launch& L, int dtype, const void* w, const void* u, const float* bias, void* v,
                   int out_dtype, const int* len_out, int B, int Cin, int Cout, int Tp) {
    KScope ks_(L, KC_PW_FWD, (double)B * Tp * (dtype_size(dtype) * Cin + dtype_size(out_dtype) * Cout), 2.0 * B * Tp * Cin * Cout);
    GemmDesc d{};
    d.M = Cout; d.N = Tp; d.Kd = Cin;
    d.a_z = 0; d.a_m = Cin; d.a_k = 1;
    d.b_z = (long long)Cin * Tp; d.b_k = Tp; d.b_n = 1;
    if (out_dtype == dtype) {
        SC_DISPATCH(dtype, (launch_gemm<T, T, 0>(L, d, B, w, u, v, bias, len_out)));
    } else if (dtype == BF16 && out_dtype == F16) {   // bfloat16 operands, float16 result
        launch_gemm<__nv_bfloat16, __half, 0>(L, d, B, w, u, v, bias, len_out);
    } else if (dtype == BF16) {   // 16-bit operands, float result
        launch_gemm<__nv_bfloat16, float, 0>(L, d, B, w, u, v, bias, len_out);
    } else {
        launch_gemm<__half, float, 0>(L, d, B, w, u, v, bias, len_out);
    }
    L.count();
}

void gemm_dgrad_simt(const Launch& L, int dtype, const void* w, const void* gv, void* gu, int B, int Cin,
                     int Cout, int Tp) {
    KScope ks_(L, KC_PW_DGRAD, (double)dtype_size(dtype) * B * Tp * (Cin + Cout), 2.0 * B * Tp * Cin * Cout);
    GemmDesc d{};
    d.M = Cin; d.N = Tp; d.Kd = Cout;
    d.a_z = 0; d.a_m = 1; d.a_k = Cin;            // A(m=c, k=o) = w[o*Cin + c]
    d.b_z = (long long)Cout * Tp; d.b_k = Tp; d.b_n = 1;
    SC_DISPATCH(dtype, (launch_gemm<T, T, 1>(L, d, B, w, gv, gu, nullptr, nullptr)));
    L.count();
}

// Slices per sample: one, unless the tiles of all samples together leave SMs idle.
static int wgrad_per_sample(int B, int Cin, int Cout) {
    const long long tiles = (long long)((Cin + 31) / 32) * ((Cout + 31) / 32) * B;
    return (int)std::min(8ll, std::max(1ll, 148 / tiles));
}

size_t gemm_wgrad_simt_scratch_bytes(int B, int Cin, int Cout) {
    return (size_t)B * wgrad_per_sample(B, Cin, Cout) * Cin * Cout * sizeof(float);
}

void gemm_wgrad_simt(const Launch& L, int dtype, const void* gv, const void* u, float* dw, float* partials,
                     int accumulate, int B, int Cin, int Cout, int Tp, const float* gmax) {
    GemmDesc d{};
    d.k_len = ((Tp + wgrad_per_sample(B, Cin, Cout) - 1) / wgrad_per_sample(B, Cin, Cout) + BK - 1) / BK * BK;
    d.per_z = (Tp + d.k_len - 1) / d.k_len;
    const int ns = B * d.per_z;
    {
    KScope ks_(L, KC_PW_WGRAD, (double)dtype_size(dtype) * B * Tp * (Cin + Cout), 2.0 * B * Tp * Cin * Cout);
    d.M = Cout; d.N = Cin; d.Kd = Tp;
    d.a_z = (long long)Cout * Tp; d.a_m = Tp; d.a_k = 1;    // A(m=o, k=t) = gv[b,o,t]
    d.b_z = (long long)Cin * Tp; d.b_n = Tp; d.b_k = 1;     // B(k=t, n=c) = u[b,c,t]
    SC_DISPATCH(dtype, (launch_gemm<T, T, 2>(L, d, ns, gv, u, partials, nullptr, nullptr)));
    L.count();
    }
    reduce_partials(L, partials, ns, (int64_t)Cin * Cout, dw, accumulate, gmax);
}

}  // namespace sc
