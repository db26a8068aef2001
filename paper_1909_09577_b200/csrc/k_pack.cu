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
    const int C = p.l.C[k], nrows = p.B * C;
    const uint32_t total = (uint32_t)nrows * p.T, f = idx * 8, total_p = (uint32_t)nrows * D * p.Tq;
    const void* src = p.l.src[k];
    unsigned short* dst = (unsigned short*)p.l.dst[k];
    const uint32_t row = p.dT.div(f);
    const int t = (int)(f - row * p.T), left = (int)min(8u, total - f);
    // frames t .. t + 7 of a row, zero past the sample's length
    auto frames = [&](uint32_t r, int t0, bool aligned) -> uint4 {
        const int b = (int)(r / C), c = (int)(r - (uint32_t)b * C);
        const int n = (p.l.len[k] ? min(p.l.len[k][b], p.T) : p.T) - t0;
        if (n <= 0) return make_uint4(0, 0, 0, 0);
        const uint4 q = Packed8<D>(src, b, c, C, p.Tq, t0, total_p, aligned).get();
        return n < 8 ? keep_first(q, n) : q;
    };
    if (p.T >= 8) {
        uint4 q = frames(row, t, (p.T & 7) == 0);
        const int own = p.T - t;
        if (own < 8 && (int)row + 1 < nrows) q = splice(q, frames(row + 1, -own, false), own);
        st8_first(dst + f, q, left);
        return;
    }
    for (uint32_t e = f; e < f + left; ++e) {
        const uint32_t r = p.dT.div(e);
        const int te = (int)(e - r * p.T), b = (int)(r / C), c = (int)(r - (uint32_t)b * C);
        const int len = p.l.len[k] ? min(p.l.len[k][b], p.T) : p.T;
        dst[e] = te < len ? ((const unsigned short*)src)[((size_t)(b * D + (D == 2 ? (te & 1) : 0)) * C + c) * p.Tq + (D == 2 ? te >> 1 : te)]
                          : (unsigned short)0;
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
