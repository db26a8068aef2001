// Shared device helpers: storage-type conversion, warp reductions, status word.
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace sc {

enum DType : int { F32 = 0, F16 = 1, BF16 = 2 };

// Device status codes (mirrors sc_status in the public header).
constexpr int kErrLengths = -8;
constexpr int kErrTimeout = -9;
constexpr int kErrRange = -12;

// Power-of-two scale that brings a tensor with the given absolute maximum into [0.5, 1).
// Multiplying by it (and later by its reciprocal) is exact.
__device__ __forceinline__ float pow2_scale(float amax) {
    if (!(amax > 0.f) || !(amax < 3.0e38f)) return 1.f;
    int e;
    frexpf(amax, &e);
    e = max(-100, min(100, e));
    return ldexpf(1.f, -e);
}
// Power-of-two scale for bfloat16 taps with the given absolute maximum that become float16 operands: the maximum comes to lie in
// [2^14, 2^15), so every tap down to 2^-31 of it keeps all of its bits (unscaled, taps below 2^-14 lost theirs).
__device__ __forceinline__ float tap_scale(float amax) { return 16384.f * 2.f * pow2_scale(amax); }
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <typename T> struct IO;
template <> struct IO<float> {
    static __device__ __forceinline__ float ld(const float* p) { return *p; }
    static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
};
template <> struct IO<__half> {
    static __device__ __forceinline__ float ld(const __half* p) { return __half2float(*p); }
    static __device__ __forceinline__ void st(__half* p, float v) { *p = __float2half_rn(v); }
};
template <> struct IO<__nv_bfloat16> {
    static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

template <typename T> __device__ __forceinline__ float ldf(const T* p) { return IO<T>::ld(p); }
template <typename T> __device__ __forceinline__ void stf(T* p, float v) { IO<T>::st(p, v); }

// Round a float through the storage type (what a store followed by a load would give).
template <typename T> __device__ __forceinline__ float round_io(float v);
template <> __device__ __forceinline__ float round_io<float>(float v) { return v; }
template <> __device__ __forceinline__ float round_io<__half>(float v) { return __half2float(__float2half_rn(v)); }
template <> __device__ __forceinline__ float round_io<__nv_bfloat16>(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// vhat = (v - mean) * invstd in exactly these two float operations wherever it is needed (forward apply,
// backward reduce and apply): the normalised value is never stored, and the ReLU decision derived from it
// must be the same bit on every path.
__device__ __forceinline__ float bn_norm(float v, float mu, float is) { return __fmul_rn(__fsub_rn(v, mu), is); }

// Two-wide fp32 arithmetic (one instruction for a pair of floats; each lane rounds like the scalar
// instruction, so a value computed here equals the one computed by the scalar helper above).
namespace pk {
__device__ __forceinline__ uint64_t pack(float a, float b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void unpack(uint64_t r, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); }
__device__ __forceinline__ uint64_t add(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t mul(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t fma(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
// (v - mu) * is for a pair: nmu = pack(-mu, -mu), is2 = pack(is, is); same bits as bn_norm on each lane
__device__ __forceinline__ uint64_t bn_norm2(uint64_t v, uint64_t nmu, uint64_t is2) { return mul(add(v, nmu), is2); }
}  // namespace pk

// Is the value, once rounded to the storage type T, greater than zero?  Rounding to nearest even sends
// everything up to half the smallest subnormal to zero, so the test is a comparison with that constant:
// the same decision as round_io<T>(a) > 0 without the two conversions.
template <typename T> __device__ __forceinline__ bool rounds_positive(float a);
template <> __device__ __forceinline__ bool rounds_positive<float>(float a) { return a > 0.f; }
template <> __device__ __forceinline__ bool rounds_positive<__half>(float a) { return a > 0x1p-25f; }
template <> __device__ __forceinline__ bool rounds_positive<__nv_bfloat16>(float a) { return a > 0x1p-134f; }

// Rounds the first n of 8 consecutive values to the storage type with error diffusion: the rounding
// residual of one element is added to the next before it is rounded, so the residuals of a vector do
// not add up.  Plain rounding is biased whenever the values sit on a lattice that the storage grid
// resolves only up to a constant offset (a 16-bit gradient times a short binary fraction, minus a
// per-channel constant); a bias of a fraction of a unit in the last place per element, summed over
// every frame of a channel by the weight-gradient contraction, would dominate that gradient's error.
template <typename ST> __device__ __forceinline__ void diffuse8(float (&v)[8], int n) {
    if (sizeof(ST) == 4) return;
    float r = 0.f;
    if (n >= 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float t = v[i] + r;
            const float q = round_io<ST>(t);
            r = t - q;
            v[i] = q;
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (i < n) {
            const float t = v[i] + r;
            const float q = round_io<ST>(t);
            r = t - q;
            v[i] = q;
        }
    }
}

// 8 consecutive elements <-> 8 floats.  Pointers must be aligned to 8 elements.
template <typename T> __device__ __forceinline__ void ld8(const T* p, float (&f)[8]);
template <> __device__ __forceinline__ void ld8<float>(const float* p, float (&f)[8]) {
    float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
template <> __device__ __forceinline__ void ld8<__half>(const __half* p, float (&f)[8]) {
    uint4 r = *reinterpret_cast<const uint4*>(p);
    const __half2* h = reinterpret_cast<const __half2*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) { float2 q = __half22float2(h[i]); f[2 * i] = q.x; f[2 * i + 1] = q.y; }
}
template <> __device__ __forceinline__ void ld8<__nv_bfloat16>(const __nv_bfloat16* p, float (&f)[8]) {
    uint4 r = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) { float2 q = __bfloat1622float2(h[i]); f[2 * i] = q.x; f[2 * i + 1] = q.y; }
}
// the same conversion from a 16-byte vector that is already in registers (16-bit types)
template <typename T> __device__ __forceinline__ void cvt8(const uint4& r, float (&f)[8]);
template <> __device__ __forceinline__ void cvt8<__half>(const uint4& r, float (&f)[8]) {
    const __half2* h = reinterpret_cast<const __half2*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) { float2 q = __half22float2(h[i]); f[2 * i] = q.x; f[2 * i + 1] = q.y; }
}
template <> __device__ __forceinline__ void cvt8<__nv_bfloat16>(const uint4& r, float (&f)[8]) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) { float2 q = __bfloat1622float2(h[i]); f[2 * i] = q.x; f[2 * i + 1] = q.y; }
}
template <typename T> __device__ __forceinline__ void st8(T* p, const float (&f)[8]);
template <> __device__ __forceinline__ void st8<float>(float* p, const float (&f)[8]) {
    *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
    *reinterpret_cast<float4*>(p + 4) = make_float4(f[4], f[5], f[6], f[7]);
}
template <> __device__ __forceinline__ void st8<__half>(__half* p, const float (&f)[8]) {
    uint4 r;
    __half2* h = reinterpret_cast<__half2*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2half2_rn(f[2 * i], f[2 * i + 1]);
    *reinterpret_cast<uint4*>(p) = r;
}
template <> __device__ __forceinline__ void st8<__nv_bfloat16>(__nv_bfloat16* p, const float (&f)[8]) {
    uint4 r;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    *reinterpret_cast<uint4*>(p) = r;
}

// Elements of a 16-byte aligned dense 16-bit array that start at any element index.  Fetching and picking are two steps, so
// that a thread can have the aligned vectors of all its operands in flight before it waits for the first (fetched and
// shifted one after the other, behind a branch on the alignment, the unaligned batch-norm kernels took 2-3 times as long as
// the aligned ones).  fetch<N>: the N aligned vectors from the one that holds element idx on; a vector past the array's last
// is replaced by the last, so no 16-byte line outside it is touched.
template <int N> struct RawVec { uint4 v[N]; };
template <int N> __device__ __forceinline__ RawVec<N> fetch(const void* base, uint32_t idx, uint32_t total) {
    const uint4* p = reinterpret_cast<const uint4*>(base);
    const uint32_t q = idx >> 3, last = (total - 1) >> 3;
    RawVec<N> r;
#pragma unroll
    for (int i = 0; i < N; ++i) r.v[i] = p[min(q + i, last)];
    return r;
}
// w[0 ..] <- w[off ..], off in 0 .. 3 (the first n words of the result are used)
template <int M> __device__ __forceinline__ void shift_words(uint32_t (&w)[M], int n, uint32_t off) {
#pragma unroll
    for (int i = 0; i < M - 2; ++i) if (i < n + 1) w[i] = (off & 2) ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < M - 3; ++i) if (i < n) w[i] = (off & 1) ? w[i + 1] : w[i];
}
// elements idx, idx + 1, ..., idx + 7
__device__ __forceinline__ uint4 pick8(const RawVec<2>& r, uint32_t idx) {
    uint32_t w[8] = {r.v[0].x, r.v[0].y, r.v[0].z, r.v[0].w, r.v[1].x, r.v[1].y, r.v[1].z, r.v[1].w};
    shift_words(w, 5, (idx >> 1) & 3);
    const uint32_t sh = (idx & 1) * 16;
    return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh), __funnelshift_r(w[2], w[3], sh),
                      __funnelshift_r(w[3], w[4], sh));
}
// elements idx, idx + 2, ..., idx + 14
__device__ __forceinline__ uint4 pick8_even(const RawVec<3>& r, uint32_t idx) {
    uint32_t w[12] = {r.v[0].x, r.v[0].y, r.v[0].z, r.v[0].w, r.v[1].x, r.v[1].y, r.v[1].z, r.v[1].w, r.v[2].x, r.v[2].y, r.v[2].z, r.v[2].w};
    shift_words(w, 8, (idx >> 1) & 3);
    const uint32_t sel = (idx & 1) ? 0x7632u : 0x5410u;
    return make_uint4(__byte_perm(w[0], w[1], sel), __byte_perm(w[2], w[3], sel), __byte_perm(w[4], w[5], sel), __byte_perm(w[6], w[7], sel));
}
__device__ __forceinline__ uint4 ld8_any(const void* base, uint32_t idx, uint32_t total) { return pick8(fetch<2>(base, idx, total), idx); }

// Eight consecutive frames t .. t + 7 of dense row (b, c) from a packed tensor [B D, C, Tq] (kernels.h): for one phase they
// are contiguous, for two they alternate between the rows of the phases, four from each (aligned when the dense rows are
// whole vectors).  t may lie up to 7 frames outside the row on either side; what is picked there is unspecified.
template <int D> struct Packed8 {
    RawVec<2> r; uint32_t idx;
    __device__ __forceinline__ Packed8() : r{}, idx(0) {}
    __device__ __forceinline__ Packed8(const void* src, int b, int c, int C, int Tq, int t, uint32_t total, bool aligned) {
        if (D == 1) { idx = ((uint32_t)b * C + c) * Tq + t; r = fetch<2>(src, idx, total); return; }
        const unsigned short* s = reinterpret_cast<const unsigned short*>(src);
        const uint32_t i0 = ((uint32_t)(b * 2 + (t & 1)) * C + c) * Tq + (t >> 1), i1 = ((uint32_t)(b * 2 + ((t + 1) & 1)) * C + c) * Tq + ((t + 1) >> 1);
        idx = 0;
        uint2 a, h;
        if (aligned) {
            a = *reinterpret_cast<const uint2*>(s + i0); h = *reinterpret_cast<const uint2*>(s + i1);
        } else {
            uint32_t e[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) { e[i] = s[min(i0 + i, total - 1)]; e[4 + i] = s[min(i1 + i, total - 1)]; }
            a = make_uint2(e[0] | (e[1] << 16), e[2] | (e[3] << 16)); h = make_uint2(e[4] | (e[5] << 16), e[6] | (e[7] << 16));
        }
        r.v[0] = make_uint4(a.x, a.y, h.x, h.y);
    }
    __device__ __forceinline__ uint4 get() const {
        if (D == 1) return pick8(r, idx);
        const uint4 q = r.v[0];
        return make_uint4(__byte_perm(q.x, q.z, 0x5410), __byte_perm(q.x, q.z, 0x7632), __byte_perm(q.y, q.w, 0x5410), __byte_perm(q.y, q.w, 0x7632));
    }
};
// zeroes the elements n, n + 1, ... (n < 8) of a vector of eight 16-bit elements
__device__ __forceinline__ uint4 keep_first(const uint4& r, int n) {
    uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (2 * i >= n) w[i] = 0u;
        else if (2 * i + 1 >= n) w[i] &= 0x0000FFFFu;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// elements [0, n) of a, the rest of b
__device__ __forceinline__ uint4 splice(const uint4& a, const uint4& b, int n) {
    uint32_t x[4] = {a.x, a.y, a.z, a.w};
    const uint32_t y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (2 * i >= n) x[i] = y[i];
        else if (2 * i + 1 >= n) x[i] = (x[i] & 0x0000FFFFu) | (y[i] & 0xFFFF0000u);
    }
    return make_uint4(x[0], x[1], x[2], x[3]);
}
// the first n elements of a 16-byte vector to p (16-byte aligned)
__device__ __forceinline__ void st8_first(unsigned short* p, const uint4& r, int n) {
    if (n >= 8) { *reinterpret_cast<uint4*>(p) = r; return; }
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) if (i < n) p[i] = (unsigned short)(w[i >> 1] >> (16 * (i & 1)));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Chan/Welford merge of (n_a, mean_a, M2_a) with (n_b, mean_b, M2_b).
__device__ __forceinline__ void chan_merge(float& n, float& mean, float& m2, float nb, float meanb, float m2b) {
    if (nb == 0.f) return;
    float nt = n + nb;
    float d = meanb - mean;
    mean += d * (nb / nt);
    m2 += m2b + d * d * (n * nb / nt);
    n = nt;
}

// Programmatic dependent launch.  Every kernel of the library is launched so that it may start while the
// kernel before it on the stream is still running.  It (1) waits for the kernels before it to complete, with their writes
// visible, before it reads or writes global memory, and (2) tells the runtime after that wait that its own dependents may
// be launched.  Work placed before pdl_wait() (barrier set-up, tensor-memory allocation, descriptor prefetch) overlaps the
// previous kernel.  Because the trigger comes after the wait, a kernel starts only once everything up to the kernel before
// the previous one has completed; so it may also read, ahead of its wait, what was settled that early: the caller's
// parameters (from the second kernel of a call on) and what the prologue wrote (such kernels go through launch_early in
// kernels.h, where the rules stand).  Both are no-ops in a kernel launched without the attribute.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_sync() { pdl_wait(); pdl_launch_dependents(); }

__device__ __forceinline__ void raise_status(int* status, int code) {
    if (status) atomicCAS(status, 0, code);
}

}  // namespace sc
