// Stride-2 depthwise correlation of 16-bit tensors (the encoder's first layer): forward, input gradient, tap gradient.
//
// With stride 2 a frame meets only the taps of one parity, so every sum splits into two correlations with adjacent taps on
// the even and the odd frames.  The tiles are de-interleaved once, on the way into shared memory, and the register blocking
// of the stride-1 kernels then applies to each half: 8 outputs and 8 taps per step, 64 multiply-adds per four 16-byte
// shared loads.  The kernels this replaces read one shared word per multiply-add (forward, with two-way bank conflicts) or
// tested every tap for its parity (input gradient).  32 samples x 64 channels x 1600 frames, K = 33, bf16:
// forward 25.1 -> 10.7 us, input gradient 201.5 -> 10.6, tap gradient 22.8 -> 9.9 (HBM time of each: 1.5 us; what is left is
// the multiply-adds, about 3 us at the fp32 peak, and the staging).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace sc {
namespace {

constexpr int R = 8;              // outputs per thread and parity
constexpr int CH = 8;             // channels (warps) per CTA
constexpr int TT = 32 * R;        // outputs per warp (forward); pairs of outputs per warp (input gradient)

// 16-byte shared loads at an 8-float lane pitch without bank conflicts
__device__ __forceinline__ int phys(int i) { return i + ((i >> 5) << 2); }
inline int host_phys(int i) { return i + ((i >> 5) << 2); }
__device__ __forceinline__ void ld_win(const float* s, int i, float* w) {
    const float4 a = *reinterpret_cast<const float4*>(s + phys(i)), b = *reinterpret_cast<const float4*>(s + phys(i + 4));
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}
__device__ __forceinline__ void ld_taps(const float* s, float* w) {
    const float4 a = *reinterpret_cast<const float4*>(s), b = *reinterpret_cast<const float4*>(s + 4);
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}

// u[t] = sum_k w[k] x[2 t + k - P].  Taps are added in the order 0, 1, 2, ... for every output, like the plain kernel's.
template <typename T, typename TO>
__global__ void __launch_bounds__(32 * CH)
dw_s2_fwd_kernel(const T* __restrict__ x, const T* __restrict__ w, TO* __restrict__ u, const int* __restrict__ len_in,
                 const int* __restrict__ len_out, int C, int Tt, int Tp, int K, int Kh, int* status) {
    extern __shared__ float smem[];
    const int lane = threadIdx.x, wrp = threadIdx.y;
    const int b = blockIdx.z, c = blockIdx.y * CH + wrp, t0 = blockIdx.x * TT;
    if (c >= C) return;                       // warps are independent
    const int P = (K - 1) / 2, XW = TT + Kh, XP = phys(XW) + 4;
    float* xe = smem + (size_t)wrp * (2 * XP + 2 * Kh);      // frames 2 t0 - P + 2 i
    float* xo = xe + XP;                                     // frames 2 t0 - P + 2 i + 1
    float* we = xo + XP;                                     // even taps, then odd taps, zero padded to Kh each
    float* wo = we + Kh;
    for (int j = lane; j < Kh; j += 32) {
        we[j] = 2 * j < K ? ldf(w + (size_t)c * K + 2 * j) : 0.f;
        wo[j] = 2 * j + 1 < K ? ldf(w + (size_t)c * K + 2 * j + 1) : 0.f;
    }
    pdl_sync();                               // the taps are the caller's parameters
    const int li = min(len_in[b], Tt), lo = min(len_out[b], Tp);
    TO* urow = u + ((size_t)b * C + c) * Tp;
    const int t = t0 + lane * R;
    if (t0 >= lo) {
        const float z[8] = {};
        if (t < Tp) st8<TO>(urow + t, z);
        return;
    }
    const T* xrow = x + ((size_t)b * C + c) * Tt;
    const int tau0 = 2 * t0 - P, a0 = tau0 & ~7;             // arithmetic: rounds towards minus infinity
    for (int ta = a0 + 8 * lane; ta < tau0 + 2 * XW; ta += 256) {
        float f[8] = {};
        if (ta >= 0 && ta < Tt) ld8<T>(xrow + ta, f);          // not bounded by li: need not wait for it
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int i = ta + e - tau0;
            if (i >= 0 && i < 2 * XW) ((i & 1) ? xo : xe)[phys(i >> 1)] = ta + e < li ? f[e] : 0.f;
        }
    }
    __syncwarp();
    float acc[R] = {}, e[2 * R], o[2 * R];
    const int base = lane * R;
    ld_win(xe, base, e); ld_win(xo, base, o);
    for (int j = 0; j < Kh; j += R) {
        float a[R], h[R];
        ld_win(xe, base + j + R, e + R); ld_win(xo, base + j + R, o + R);
        ld_taps(we + j, a); ld_taps(wo + j, h);
#pragma unroll
        for (int q = 0; q < R; ++q) {
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fmaf(a[q], e[r + q], acc[r]);
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fmaf(h[q], o[r + q], acc[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) { e[r] = e[r + R]; o[r] = o[r + R]; }
    }
    if (t >= Tp) return;
    bool over = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (std::is_same<TO, __half>::value && fabsf(acc[r]) > 65504.f) { acc[r] = copysignf(65504.f, acc[r]); over = true; }
        if (t + r >= lo) acc[r] = 0.f;
    }
    if (over) raise_status(status, kErrRange);
    st8<TO>(urow + t, acc);
}

// dx[tau] = sum over the taps k with tau + P - k even of w[k] gu[(tau + P - k) / 2].  The outputs with tau + P = 2 a + e
// take the taps 2 j + e and gu[a - j]: a thread owns 16 consecutive outputs, eight of each parity, on one window of gu.
// OP = P & 1: then the even-tap outputs sit one gu frame later than the odd-tap ones.
template <typename TG, typename T, int OP>
__global__ void __launch_bounds__(32 * CH)
dw_s2_dgrad_kernel(const TG* __restrict__ gu, const T* __restrict__ w, T* __restrict__ dx, const T* __restrict__ add1,
                   const T* __restrict__ add2, const float* __restrict__ gmax, const int* __restrict__ len_in,
                   const int* __restrict__ len_out, int C, int Tt, int Tp, int K, int Kh) {
    extern __shared__ float smem[];
    const int lane = threadIdx.x, wrp = threadIdx.y;
    const int b = blockIdx.z, c = blockIdx.y * CH + wrp, i0 = blockIdx.x * TT;     // output pairs i0 ..: frames 2 i, 2 i + 1
    if (c >= C) return;
    const int P = (K - 1) / 2, GW = TT + Kh + 8, GP = phys(GW) + 4;
    float* g = smem + (size_t)wrp * (GP + 2 * Kh);           // frame g0 + i
    float* we = g + GP;                                      // taps 2 (Kh - 1 - j), then 2 (Kh - 1 - j) + 1
    float* wo = we + Kh;
    for (int j = lane; j < Kh; j += 32) {
        const int k = 2 * (Kh - 1 - j);
        we[j] = k < K ? ldf(w + (size_t)c * K + k) : 0.f;
        wo[j] = k + 1 < K ? ldf(w + (size_t)c * K + k + 1) : 0.f;
    }
    pdl_sync();
    const int li = min(len_in[b], Tt), lo = min(len_out[b], Tp);
    const size_t row = ((size_t)b * C + c) * Tt;
    const int tau = 2 * i0 + 16 * lane;
    if (2 * i0 >= li) {
        const float z[8] = {};
        if (tau < Tt) { st8<T>(dx + row + tau, z); st8<T>(dx + row + tau + 8, z); }
        return;
    }
    // odd-tap outputs of pair i: a = i + P / 2; even-tap ones: a + OP; the first frame met is a - (Kh - 1)
    const int g0 = i0 + P / 2 - (Kh - 1), a0 = g0 & ~7;
    const TG* grow = gu + ((size_t)b * C + c) * Tp;
    for (int ta = a0 + 8 * lane; ta < g0 + GW; ta += 256) {
        float f[8] = {};
        if (ta >= 0 && ta < lo) ld8<TG>(grow + ta, f);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int i = ta + e - g0;
            if (i >= 0 && i < GW) g[phys(i)] = ta + e < lo ? f[e] : 0.f;
        }
    }
    __syncwarp();
    float ae[R] = {}, ao[R] = {}, win[2 * R];
    const int base = lane * R;
    ld_win(g, base, win); ld_win(g, base + R, win + R);
    for (int j = 0; j < Kh; j += R) {
        float a[R], h[R];
        ld_taps(we + j, a); ld_taps(wo + j, h);
#pragma unroll
        for (int q = 0; q < R; ++q) {
#pragma unroll
            for (int r = 0; r < R; ++r) ae[r] = fmaf(a[q], win[r + q + OP], ae[r]);
#pragma unroll
            for (int r = 0; r < R; ++r) ao[r] = fmaf(h[q], win[r + q], ao[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) win[r] = win[r + R];
        ld_win(g, base + j + 2 * R, win + R);
    }
    if (tau >= Tt) return;
    const float inv = gmax ? 1.f / pow2_scale(*gmax) : 1.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float f[8];
#pragma unroll
        for (int r = 0; r < 4; ++r) {          // P even: frame 2 i meets the even taps; P odd: the odd ones
            f[2 * r] = (OP ? ao : ae)[4 * h + r] * inv;
            f[2 * r + 1] = (OP ? ae : ao)[4 * h + r] * inv;
        }
        const int t = tau + 8 * h;
        if (add1) { float q[8]; ld8<T>(add1 + row + t, q);
#pragma unroll
            for (int r = 0; r < 8; ++r) f[r] += q[r]; }
        if (add2) { float q[8]; ld8<T>(add2 + row + t, q);
#pragma unroll
            for (int r = 0; r < 8; ++r) f[r] += q[r]; }
#pragma unroll
        for (int r = 0; r < 8; ++r) if (t + r >= li) f[r] = 0.f;
        st8<T>(dx + row + t, f);
    }
}

// dwd[k] = sum_{b,t} gu[t] x[2 t + k - P].  The de-interleaved rows of x stay 16-bit in shared memory (H zeros in front),
// and tap k is offset m = H + floor((k - P) / 2) of its parity's row.  A thread owns 8 frames of gu and every offset:
// 16 NCH accumulators, two 16-wide windows.  Sums go over the warp by halving exchange, then over the warps in order.
constexpr int WT = 128;           // threads
constexpr int WTT = 1024;         // frames of gu per stage

template <typename TG, typename T, int NCH>
__global__ void __launch_bounds__(WT)
dw_s2_wgrad_kernel(const TG* __restrict__ gu, const T* __restrict__ x, float* __restrict__ partials, const int* __restrict__ len_in,
                   const int* __restrict__ len_out, int B, int C, int Tt, int Tp, int K, int H, int per) {
    pdl_sync();
    constexpr int XW = WTT + 8 * NCH + 8;                    // a window reads up to offset 8 NCH + 7 past its frame
    __shared__ __align__(16) unsigned short gs[WTT];
    __shared__ __align__(16) unsigned short xs[2][XW];
    __shared__ float red[WT / 32][16 * NCH];
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wrp = tid >> 5;
    const int P = (K - 1) / 2;
    float acc[2][8 * NCH];
#pragma unroll
    for (int i = 0; i < 8 * NCH; ++i) acc[0][i] = acc[1][i] = 0.f;
    const int b1 = min(B, (int)(blockIdx.y + 1) * per);
    for (int b = blockIdx.y * per; b < b1; ++b) {
        const int li = min(len_in[b], Tt), lo = min(len_out[b], Tp);
        const TG* grow = gu + ((size_t)b * C + c) * Tp;
        const T* xrow = x + ((size_t)b * C + c) * Tt;
        for (int t0 = 0; t0 < lo; t0 += WTT) {
            __syncthreads();
            const int n = min(WTT, lo - t0), nv = (n + 7) / 8;
            for (int v = tid; v < nv; v += WT) {
                uint4 r = *reinterpret_cast<const uint4*>(grow + t0 + 8 * v);
                if (8 * v + 8 > n) r = keep_first(r, n - 8 * v);
                *reinterpret_cast<uint4*>(gs + 8 * v) = r;
            }
            // rows entry i holds pair q = t0 - H + i; four pairs per 16-byte vector of x
            const int width = 8 * nv + 8 * NCH;
            for (int i = 4 * tid; i < width; i += 4 * WT) {
                const int tau = 2 * (t0 - H + i);            // a multiple of 8: H and i are multiples of 4
                uint4 r = make_uint4(0, 0, 0, 0);
                if (tau >= 0 && tau < li) {
                    r = *reinterpret_cast<const uint4*>(xrow + tau);
                    if (tau + 8 > li) r = keep_first(r, li - tau);
                }
                *reinterpret_cast<uint2*>(&xs[0][i]) = make_uint2(__byte_perm(r.x, r.y, 0x5410), __byte_perm(r.z, r.w, 0x5410));
                *reinterpret_cast<uint2*>(&xs[1][i]) = make_uint2(__byte_perm(r.x, r.y, 0x7632), __byte_perm(r.z, r.w, 0x7632));
            }
            __syncthreads();
            for (int v = tid; v < nv; v += WT) {
                float g[8];
                cvt8<TG>(*reinterpret_cast<const uint4*>(gs + 8 * v), g);
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const unsigned short* xp = xs[p] + 8 * v;
                    float win[16];
                    { float q[8]; cvt8<T>(*reinterpret_cast<const uint4*>(xp), q);
#pragma unroll
                      for (int i = 0; i < 8; ++i) win[i] = q[i]; }
#pragma unroll
                    for (int ch = 0; ch < NCH; ++ch) {
                        float q[8];
                        // the last window's upper half only meets offsets past 8 NCH - 1, except its first seven frames
                        cvt8<T>(*reinterpret_cast<const uint4*>(xp + 8 * ch + 8), q);
#pragma unroll
                        for (int i = 0; i < 8; ++i) win[8 + i] = q[i];
#pragma unroll
                        for (int m = 0; m < 8; ++m)
#pragma unroll
                            for (int r = 0; r < 8; ++r) acc[p][8 * ch + m] = fmaf(g[r], win[r + m], acc[p][8 * ch + m]);
#pragma unroll
                        for (int i = 0; i < 8; ++i) win[i] = win[8 + i];
                    }
                }
            }
        }
    }
    // Lane pairs split the live values between them, each keeps one half and adds the partner's copy of it.
    constexpr int VP = (16 * NCH + 31) / 32 * 32;
    float v[VP];
#pragma unroll
    for (int i = 0; i < VP; ++i) v[i] = i < 8 * NCH ? acc[0][i] : (i < 16 * NCH ? acc[1][i - 8 * NCH] : 0.f);
    int base = 0;
#pragma unroll
    for (int s = 16, n = VP / 2; s >= 1; s >>= 1, n >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float lo = v[i], hi = v[i + n];
            const float got = __shfl_xor_sync(0xffffffffu, up ? lo : hi, s);
            v[i] = (up ? hi : lo) + got;
        }
        if (up) base += n;
    }
#pragma unroll
    for (int i = 0; i < VP / 32; ++i) if (base + i < 16 * NCH) red[wrp][base + i] = v[i];
    __syncthreads();
    for (int k = tid; k < K; k += WT) {
        const int d = k - P, m = H + (d >> 1) + ((d & 1) ? 8 * NCH : 0);      // d >> 1 rounds down; odd d: the odd row
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < WT / 32; ++q) s += red[q][m];
        partials[((size_t)blockIdx.y * C + c) * K + k] = s;
    }
}

int half_taps(int K) { return ((K + 1) / 2 + R - 1) / R * R; }
int lead(int K) { return (((K - 1) / 2 + 1) / 2 + 3) / 4 * 4; }           // H: ceil(P / 2) rounded up to 4
int chunks(int K) { return (lead(K) + (K - 1) / 4 + 1 + 7) / 8; }         // NCH: offsets 0 .. H + P / 2

}  // namespace

#define SC_DISPATCH_S2(dtype, odt, ...)                                                     \
    if (dtype == F16) { using T = __half; using OT = __half; __VA_ARGS__; }                  \
    else if (odt == F16) { using T = __nv_bfloat16; using OT = __half; __VA_ARGS__; }        \
    else { using T = __nv_bfloat16; using OT = __nv_bfloat16; __VA_ARGS__; }

// rows of whole vectors on both sides; more taps than 95 would need more accumulators than a thread has registers for
bool dw_s2_supported(int dtype, int Tt, int Tp, int K) {
    return dtype != F32 && Tt == 2 * Tp && Tp % 8 == 0 && (K & 1) && chunks(K) <= 6;
}

void dw_s2_fwd(const Launch& L, int dtype, int odt, const void* x, const void* wd, void* u, const int* len_in, const int* len_out,
               int B, int C, int Tt, int Tp, int K) {
    const int Kh = half_taps(K);
    const size_t smem = (size_t)CH * (2 * (host_phys(TT + Kh) + 4) + 2 * Kh) * sizeof(float);
    const dim3 grid((Tp + TT - 1) / TT, (C + CH - 1) / CH, B), block(32, CH);
    SC_DISPATCH_S2(dtype, odt, (launch_k(L, dw_s2_fwd_kernel<T, OT>, grid, block, smem, (const T*)x, (const T*)wd, (OT*)u, len_in, len_out,
                                         C, Tt, Tp, K, Kh, L.status)));
    L.count();
}

void dw_s2_dgrad(const Launch& L, int dtype, int odt, const void* gu, const void* wd, void* dx, const void* add1, const void* add2,
                 const float* gmax, const int* len_in, const int* len_out, int B, int C, int Tt, int Tp, int K) {
    const int Kh = half_taps(K);
    const size_t smem = (size_t)CH * (host_phys(TT + Kh + 8) + 4 + 2 * Kh) * sizeof(float);
    const dim3 grid((Tp + TT - 1) / TT, (C + CH - 1) / CH, B), block(32, CH);
    if (((K - 1) / 2) & 1) {
        SC_DISPATCH_S2(dtype, odt, (launch_k(L, dw_s2_dgrad_kernel<OT, T, 1>, grid, block, smem, (const OT*)gu, (const T*)wd, (T*)dx,
                                             (const T*)add1, (const T*)add2, gmax, len_in, len_out, C, Tt, Tp, K, Kh)));
    } else {
        SC_DISPATCH_S2(dtype, odt, (launch_k(L, dw_s2_dgrad_kernel<OT, T, 0>, grid, block, smem, (const OT*)gu, (const T*)wd, (T*)dx,
                                             (const T*)add1, (const T*)add2, gmax, len_in, len_out, C, Tt, Tp, K, Kh)));
    }
    L.count();
}

// returns the number of partial rows [C, K] written
int dw_s2_wgrad(const Launch& L, int dtype, int odt, const void* gu, const void* x, float* partials, const int* len_in,
                const int* len_out, int B, int C, int Tt, int Tp, int K) {
    // about 600 CTAs (four per SM) where the batch has that many samples
    const int per = std::max(1, (int)((long long)B * C / 600)), ns = (B + per - 1) / per, H = lead(K);
    const dim3 grid(C, ns);
#define SC_S2_CASE(N) case N: SC_DISPATCH_S2(dtype, odt, (launch_k(L, dw_s2_wgrad_kernel<OT, T, N>, grid, WT, 0, (const OT*)gu, (const T*)x, \
                                             partials, len_in, len_out, B, C, Tt, Tp, K, H, per))) break;
    switch (chunks(K)) { SC_S2_CASE(1) SC_S2_CASE(2) SC_S2_CASE(3) SC_S2_CASE(4) SC_S2_CASE(5) SC_S2_CASE(6) }
#undef SC_S2_CASE
    return ns;              // the caller counts the launch
}

}  // namespace sc
