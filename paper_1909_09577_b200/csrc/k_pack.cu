// Copies between dense [B, C, T] tensors of any row length and the packed form that the tensor-core kernels read
// (kernels.h, "packed tensors").  16-bit elements; pure data movement, bound by HBM / L2 bandwidth: every thread moves
// whole 16-byte vectors on both sides (a vector that starts anywhere in a row is two aligned loads and a funnel shift),
// and up to kMaxPack tensors share one launch.
// What packing buys (B200, forward + backward of one block, before: plain SIMT kernels on the dense tensors): bf16 384 -> 384,
// K = 39, 23 samples of 797 frames with the projected residual 2084 -> 297 us; 512 -> 512, K = 87, dilation 2, 16 samples of
// 800 frames 1629 -> 180 us.  A copy of 16 MB takes 5-10 us.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace sc {
namespace {

struct PackArgs { PackList l; int B, T, Tq; FastDiv dvpr, dT; uint32_t nvec[kMaxPack]; };

// one packed 16-byte vector per thread (D = 2: the same vector position of both phases)
template <int D>
__global__ void __launch_bounds__(256) pack_kernel(PackArgs p) {
    pdl_sync();
    const int k = blockIdx.y;
    const uint32_t idx = blockIdx.x * 256u + threadIdx.x;
    if (idx >= p.nvec[k]) return;
    const int vpr = p.Tq / 8, C = p.l.C[k];
    const uint32_t row = p.dvpr.div(idx);                  // dense row
    const int q0 = (int)(idx - row * vpr) * 8;
    const int b = (int)(row / C), c = (int)(row - (uint32_t)b * C);
    const int len = p.l.len[k] ? min(p.l.len[k][b], p.T) : p.T;
    const uint32_t total = (uint32_t)p.B * C * p.T;
    const void* src = p.l.src[k];
    unsigned short* dst = (unsigned short*)p.l.dst[k];
    if (D == 1) {
        const int n = len - q0;
        uint4 r = make_uint4(0, 0, 0, 0);
        if (n > 0) { r = ld8_any(src, row * p.T + q0, total); if (n < 8) r = keep_first(r, n); }
        *reinterpret_cast<uint4*>(dst + (size_t)row * p.Tq + q0) = r;
    } else {
        const int n = len - 2 * q0;                        // dense frames left
        uint4 a = make_uint4(0, 0, 0, 0), h = a;
        if (n > 0) { a = ld8_any(src, row * p.T + 2 * q0, total); if (n < 8) a = keep_first(a, n); }
        if (n > 8) { h = ld8_any(src, row * p.T + 2 * q0 + 8, total); if (n < 16) h = keep_first(h, n - 8); }
        const size_t o0 = ((size_t)(2 * b) * C + c) * p.Tq + q0, o1 = o0 + (size_t)C * p.Tq;
        *reinterpret_cast<uint4*>(dst + o0) = make_uint4(__byte_perm(a.x, a.y, 0x5410), __byte_perm(a.z, a.w, 0x5410),
                                                         __byte_perm(h.x, h.y, 0x5410), __byte_perm(h.z, h.w, 0x5410));
        *reinterpret_cast<uint4*>(dst + o1) = make_uint4(__byte_perm(a.x, a.y, 0x7632), __byte_perm(a.z, a.w, 0x7632),
                                                         __byte_perm(h.x, h.y, 0x7632), __byte_perm(h.z, h.w, 0x7632));
    }
}

// one aligned 16-byte vector of the dense tensor per thread
template <int D>
__global__ void __launch_bounds__(256) unpack_kernel(PackArgs p) {
    pdl_sync();
    const int k = blockIdx.y;
    const uint32_t idx = blockIdx.x * 256u + threadIdx.x;
    if (idx >= p.nvec[k]) return;
    const int C = p.l.C[k];
    const uint32_t total = (uint32_t)p.B * C * p.T, f = idx * 8;
    const unsigned short* src = (const unsigned short*)p.l.src[k];
    unsigned short* dst = (unsigned short*)p.l.dst[k];
    const uint32_t row = p.dT.div(f);
    const int t = (int)(f - row * p.T);
    const int b = (int)(row / C), c = (int)(row - (uint32_t)b * C);
    if (D == 1 && t + 8 <= p.T && f + 8 <= total) {
        const int n = (p.l.len[k] ? min(p.l.len[k][b], p.T) : p.T) - t;
        uint4 r = make_uint4(0, 0, 0, 0);
        if (n > 0) { r = ld8_any(src, row * p.Tq + t, (uint32_t)p.B * C * p.Tq); if (n < 8) r = keep_first(r, n); }
        *reinterpret_cast<uint4*>(dst + f) = r;
        return;
    }
    unsigned short h[8];
    int bb = b, cc = c, tt = t;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        h[i] = 0;
        if (f + i < total) {
            const int len = p.l.len[k] ? min(p.l.len[k][bb], p.T) : p.T;
            if (tt < len) h[i] = src[((size_t)(bb * D + (D == 2 ? (tt & 1) : 0)) * C + cc) * p.Tq + (D == 2 ? tt >> 1 : tt)];
            if (++tt == p.T) { tt = 0; if (++cc == C) { cc = 0; ++bb; } }
        }
    }
    if (f + 8 <= total) {
        *reinterpret_cast<uint4*>(dst + f) = make_uint4(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16),
                                                        h[4] | ((uint32_t)h[5] << 16), h[6] | ((uint32_t)h[7] << 16));
    } else {
        for (int i = 0; i < 8; ++i) if (f + i < total) dst[f + i] = h[i];
    }
}

}  // namespace

void pack_frames(const Launch& L, const PackList& list, int B, int T, int Tq, int phases) {
    if (list.count == 0) return;
    PackArgs p{}; p.l = list; p.B = B; p.T = T; p.Tq = Tq;
    p.dvpr = FastDiv((uint32_t)(Tq / 8));
    uint32_t most = 0; double bytes = 0;
    for (int k = 0; k < list.count; ++k) {
        p.nvec[k] = (uint32_t)B * list.C[k] * (Tq / 8);
        most = std::max(most, p.nvec[k]); bytes += 2.0 * B * list.C[k] * (T + (double)Tq * phases);
    }
    KScope ks_(L, KC_EW, bytes, 0.0);
    const dim3 grid((most + 255) / 256, list.count);
    if (phases == 2) launch_k(L, pack_kernel<2>, grid, 256, 0, p);
    else launch_k(L, pack_kernel<1>, grid, 256, 0, p);
    L.count();
}

void unpack_frames(const Launch& L, const PackList& list, int B, int T, int Tq, int phases) {
    if (list.count == 0) return;
    PackArgs p{}; p.l = list; p.B = B; p.T = T; p.Tq = Tq;
    p.dT = FastDiv((uint32_t)T);
    uint32_t most = 0; double bytes = 0;
    for (int k = 0; k < list.count; ++k) {
        p.nvec[k] = ((uint32_t)B * list.C[k] * T + 7) / 8;
        most = std::max(most, p.nvec[k]); bytes += 2.0 * B * list.C[k] * (T + (double)Tq * phases);
    }
    KScope ks_(L, KC_EW, bytes, 0.0);
    const dim3 grid((most + 255) / 256, list.count);
    if (phases == 2) launch_k(L, unpack_kernel<2>, grid, 256, 0, p);
    else launch_k(L, unpack_kernel<1>, grid, 256, 0, p);
    L.count();
}

}  // namespace sc
