// C-ABI layer: argument validation, workspace planning and the launch sequence of one block and of
// the whole encoder.  All arithmetic lives in the kernel files; this file only orders launches.
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/sepconv.h"
#include "api_internal.h"
#include "common.cuh"
#include "graph_cache.h"
#include "kernels.h"
#include "tc_gemm.h"

using namespace sc;

struct sc_ctx {
    int device = 0;
    int sm_count = 0;
    int* status_dev = nullptr;
    int64_t launches = 0;
    int gemm_mode = 0;
    TcState tc;
    Prof prof;
    // A second, library-owned stream: kernels that are off the critical path of a layer (weight gradients, the
    // residual projection's contraction) run there, forked from and joined back into the caller's stream with
    // events, so that they fill the SMs a latency-bound kernel of the critical path leaves idle.
    cudaStream_t side = nullptr;
    cudaEvent_t ev[8] = {};     // backward fork (and the tap gradients' of a block call), done[0], done[1], forward fork, forward join, done[2], (unused)
    int overlap = 1;
    int pdl = 1;          // launch kernels with programmatic stream serialization
    bool fresh[2] = {};   // see launch_early in kernels.h
    GraphCache graphs;
    CallKey key;
};

namespace sc {
int ctx_device(const sc_ctx* ctx) { return ctx ? ctx->device : -1; }
const char* kclass_name(int c) {
    static const char* n[KC_COUNT] = {"lengths", "dw_fwd", "dw_dgrad", "dw_wgrad", "pw_fwd", "pw_dgrad", "pw_wgrad",
                                      "bn_stats", "bn_finalize", "bn_apply", "bn_bwd_reduce", "bn_bwd_finalize",
                                      "bn_bwd_apply", "elementwise", "reduce_partials"};
    return (c >= 0 && c < KC_COUNT) ? n[c] : "?";
}
}  // namespace sc

namespace {

size_t esize(int dtype) { return dtype == SC_F32 ? 4 : 2; }

// Bump allocator over the caller's workspace; with base == nullptr it only measures.
struct Bump {
    char* base; size_t off = 0, cap;
    Bump(void* b, size_t c) : base((char*)b), cap(c) {}
    void* take(size_t bytes) {
        size_t o = (off + 255) & ~(size_t)255;
        off = o + bytes;
        return base ? base + o : nullptr;
    }
    bool ok() const { return base == nullptr || off <= cap; }
};

struct Dims { int B, Cin, Cout, Cres, T, Tp, K, s, dil; bool plain, full; };   // plain: odd K, adjacent taps; full: non-separable convolution

int desc_dims(const sc_block_desc* d, Dims* o) {
    if (!d) return SC_ERR_NULL;
    if (d->io_dtype < 0 || d->io_dtype > 2) return SC_ERR_INCOMPATIBLE;
    if (d->B < 1 || d->C_in < 1 || d->C_out < 1 || d->T_in < 1) return SC_ERR_DIM_INCOMPATIBLE;
    o->B = d->B; o->Cin = d->C_in; o->Cout = d->C_out; o->T = d->T_in;
    o->full = d->full_conv != 0;
    if (o->full && (d->has_dw || d->log_softmax)) return SC_ERR_UNSUPPORTED;
    const bool taps = d->has_dw || o->full;       // the K-tap step: depthwise, or the non-separable convolution
    o->K = taps ? d->K : 1; o->s = taps ? d->stride : 1;
    o->dil = (taps && d->dilation > 1) ? d->dilation : 1;
    if (d->dilation < 0 || o->K < 1) return SC_ERR_UNSUPPORTED;
    if (o->s != 1 && o->s != 2) return SC_ERR_UNSUPPORTED;
    o->plain = o->dil == 1 && (o->K & 1);
    o->Tp = (o->T - 1) / o->s + 1;            // "same" padding: dil * (K - 1) zeros in total
    o->Cres = d->C_res > 0 ? d->C_res : d->C_in;
    if (d->residual < 0 || d->residual > 2) return SC_ERR_UNSUPPORTED;
    if (d->residual == SC_RES_IDENTITY && o->Cres != o->Cout) return SC_ERR_UNSUPPORTED;
    if (d->residual != SC_RES_NONE && !d->has_bn) return SC_ERR_UNSUPPORTED;
    if (!d->has_bn && d->has_relu) return SC_ERR_UNSUPPORTED;
    if (d->has_bn && d->has_bias) return SC_ERR_UNSUPPORTED;   // a bias before batch norm cancels
    if (d->log_softmax && (d->has_bn || d->has_relu || d->residual != SC_RES_NONE)) return SC_ERR_UNSUPPORTED;
    return SC_OK;
}

// Blocks that the tensor-core kernels can only take in packed form (kernels.h): a row length that is not a multiple of 8
// frames, or taps two frames apart.  The batch-norm kernels convert between the dense tensors of the call and the packed
// operands on the way; only the input, its gradient and u need a copy of their own.
struct Packed { int phases = 0, Tq = 0; Dims m; };     // m: the block on the packed operands
Packed plan_packed(const sc_block_desc* d, const Dims& m) {
    Packed k;
    if (d->io_dtype == SC_F32 || !d->has_bn || !d->has_relu || !d->res_before_relu) return k;
    if (m.full && (m.s != 1 || m.Cout % 8)) return k;       // the non-separable convolution takes any dilation as it is
    const bool dilated = !m.full && m.dil == 2 && (m.K & 1) && m.s == 1;
    if (m.dil != 1 && !dilated && !m.full) return k;
    if (!dilated && m.T % 8 == 0 && m.Tp % 8 == 0) return k;
    if (m.Cin % 8 || (d->residual == SC_RES_PROJ && m.Cres % 8)) return k;
    const int ph = dilated ? 2 : 1;
    const int Tq = dilated ? ((m.T + 1) / 2 + 7) / 8 * 8 : (m.T + 8 * m.s - 1) / (8 * m.s) * (8 * m.s);
    const long long most = (long long)m.B * ph * std::max(std::max(m.Cin, m.Cout), m.Cres) * Tq;
    if (most >= (1ll << 31)) return k;                      // the copies index with 32 bits
    k.phases = ph; k.Tq = Tq; k.m = m;
    k.m.B = m.B * ph; k.m.T = Tq; k.m.Tp = Tq / m.s; if (dilated) k.m.dil = 1; k.m.plain = (m.K & 1) != 0;
    return k;
}

int check_tensor(const sc_tensor* t, int dtype, int64_t B, int64_t C, int64_t T) {
    if (!t || !t->ptr) return SC_ERR_NULL;
    if (t->dtype != dtype || t->rank != 3) return SC_ERR_INCOMPATIBLE;
    const int64_t want[3] = {B, C, T};
    const int wtag[3] = {SC_AX_BATCH, SC_AX_CHANNEL, SC_AX_TIME};
    bool tags_ok = true, sizes_ok = true;
    for (int i = 0; i < 3; ++i) { tags_ok &= (t->tag[i] == wtag[i]); sizes_ok &= (t->size[i] == want[i]); }
    if (!tags_ok) {
        // same axes in another order -> transposed; otherwise not a [batch, channel, time] tensor
        int seen = 0;
        for (int i = 0; i < 3; ++i) if (t->tag[i] >= 0 && t->tag[i] <= 2) seen |= 1 << t->tag[i];
        return seen == 7 ? SC_ERR_TRANSPOSED : SC_ERR_INCOMPATIBLE;
    }
    if (!sizes_ok) return SC_ERR_DIM_INCOMPATIBLE;
    if (t->stride[2] != 1 || t->stride[1] != T || t->stride[0] != C * T) return SC_ERR_TRANSPOSED;
    if (((uintptr_t)t->ptr & 15) != 0) return SC_ERR_ALIGNMENT;
    return SC_OK;
}

struct BlockIO {                 // raw pointers after validation
    const void* x; const void* xres; void* y;
    const int* len_in; int* len_out; int* nvalid; int* blk_off;
    bool x_clean, res_clean;     // inputs known to be zero in padded frames
    bool lengths_ready;          // len_out / nvalid already computed
    const void* w16;             // float16 copy of wp, where the layer's operands are float16 and wp is not
    // packed block: x (and a projected xres) are packed, y and an identity xres are dense [., ., Td] with lengths
    // len_dense, and u, v, vr are also written to the dense tensors of `dense` (nullable members)
    int phases, Td; const int* len_dense; sc_block_saved dense;
};

// Type of the library-internal contraction operands (u, gv, gu) of this layer.
int op_dtype(const sc_block_desc* d) { return otype_of(d->io_dtype, d->has_dw && d->has_bn); }

// ---- forward scratch ---------------------------------------------------------------------------
struct FwdScratch { void* partials; void* partials_r; void *xr, *w16, *x_tm, *taps; float* zf32; int* len_out; int* nvalid; int* blk_off; };

bool conv_on_tc(const TcState* tc, const sc_block_desc* d, const Dims& m) {
    return m.full && tc_conv_supported(tc, d->io_dtype, m.B, m.Cin, m.Cout, m.T, m.s);
}

// copies: whether the non-separable convolution may take the operand copies of its tensor-core form; without them it runs on
// the dense tensors
void plan_fwd(const sc_block_desc* d, const Dims& m, Bump& ws, FwdScratch* f, const TcState* tc, bool copies = true) {
    f->len_out = (int*)ws.take(sizeof(int) * m.B);
    f->nvalid = (int*)ws.take(sizeof(int));
    f->blk_off = (int*)ws.take(sizeof(int) * (m.B + 1));
    f->partials = ws.take(tc_stats_bytes(m.B, m.Cout, m.Tp));
    f->partials_r = (d->residual == SC_RES_PROJ) ? ws.take(tc_stats_bytes(m.B, m.Cout, m.Tp)) : nullptr;
    f->zf32 = d->log_softmax ? (float*)ws.take(sizeof(float) * m.B * m.Cout * m.Tp) : nullptr;
    f->xr = (d->residual == SC_RES_PROJ) ? ws.take(esize(d->io_dtype) * m.B * m.Cres * m.Tp) : nullptr;
    const bool conv = copies && conv_on_tc(tc, d, m);
    f->x_tm = conv ? ws.take((size_t)2 * m.B * m.Cin * m.T) : nullptr;
    f->taps = conv ? ws.take((size_t)2 * m.Cin * m.Cout * m.K) : nullptr;
    f->w16 = (op_dtype(d) != d->io_dtype) ? ws.take((size_t)2 * m.Cout * m.Cin) : nullptr;
}

// Batch statistics of v from what the contraction left behind (or from v itself).
void finalize_stats(const Launch& L, const sc_block_desc* d, const Dims& m, StatsLayout sl, const void* v, int vdt, const int* len_out,
                    const int* nvalid, const int* blk_off, void* partials, float* mean, float* invstd, float* rmean, float* rvar) {
    if (sl.kind == 2) {
        bn_finalize_flat(L, (const float4*)partials, sl.grid, sl.tiles_m, sl.rows_per_tile, blk_off, nvalid, m.B, m.Cout,
                         d->bn_eps, d->bn_momentum, mean, invstd, rmean, rvar);
        return;
    }
    if (sl.kind == 0) { bn_stats(L, vdt, v, len_out, m.B, m.Cout, m.Tp, (float2*)partials); sl.parts_per_b = 1; sl.tile_w = m.Tp; }
    bn_finalize(L, (const float2*)partials, sl.parts_per_b, sl.tile_w, len_out, nvalid, m.B, m.Cout, d->bn_eps, d->bn_momentum,
                mean, invstd, rmean, rvar);
}

bool apply_takes_stats(int dt, const ApplyArgs& a, const StatsLayout& sl) {
    return sl.kind == 2 ? bn_apply_takes_stats(dt, a) : sl.kind == 0 && bn_small(dt, a.B, a.C, a.Tp);
}

// v = w * u for every sample (stored once, in the type it is kept in for the backward pass), plus masked
// batch statistics, unless the apply step takes them (apply: its arguments, null when it must not): then *left is what the
// contraction left behind.
void pointwise_bn(sc_ctx* ctx, const Launch& L, const sc_block_desc* d, const Dims& m, int Cin, int opdt,
                  const void* w, const void* u, void* v, const int* len_out, const int* nvalid, const int* blk_off,
                  float* mean, float* invstd, void* partials, float* rmean, float* rvar, const ApplyArgs* apply = nullptr,
                  StatsLayout* left = nullptr) {
    const int vdt = ntype_of(d->io_dtype);
    StatsLayout sl;
    if (ctx->gemm_mode == 0 && tc_fwd_supported(&ctx->tc, opdt, Cin, m.Cout, m.Tp))
        tc_gemm_fwd(&ctx->tc, L, opdt, w, u, nullptr, v, vdt, len_out, blk_off, m.B, Cin, m.Cout, m.Tp, partials, &sl);
    else
        gemm_fwd_simt(L, opdt, w, u, nullptr, v, vdt, len_out, m.B, Cin, m.Cout, m.Tp);
    if (apply && apply_takes_stats(d->io_dtype, *apply, sl)) *left = sl;
    else finalize_stats(L, d, m, sl, v, vdt, len_out, nvalid, blk_off, partials, mean, invstd, rmean, rvar);
}

// The launch context of the side stream (same status word, counters and profile), or L itself when overlap is off.
Launch side_launch(sc_ctx* ctx, const Launch& L) {
    Launch s = L;
    if (ctx->overlap && ctx->side) { s.stream = ctx->side; s.lane = 1; }
    return s;
}
// side stream waits for everything enqueued on L.stream so far
void fork_to_side(sc_ctx* ctx, const Launch& L, cudaEvent_t ev) {
    if (!(ctx->overlap && ctx->side)) return;
    cudaEventRecord(ev, L.stream);
    cudaStreamWaitEvent(ctx->side, ev, 0);
    ctx->fresh[1] = ctx->fresh[0];      // what is launched there next follows the last kernel of the caller's stream
}
void record_side(sc_ctx* ctx, cudaEvent_t ev) { if (ctx->overlap && ctx->side) cudaEventRecord(ev, ctx->side); }
void wait_side(sc_ctx* ctx, const Launch& L, cudaEvent_t ev) { if (ctx->overlap && ctx->side) cudaStreamWaitEvent(L.stream, ev, 0); }

// Evaluation mode: fixed running statistics take the place of the batch statistics.
struct InferStats { const float *mean, *var, *mean_r, *var_r; };

// v = w * u without statistics (evaluation mode); invstd <- 1 / sqrt(var + eps)
void pointwise_fixed(sc_ctx* ctx, const Launch& L, const sc_block_desc* d, const Dims& m, int Cin, int opdt, const void* w,
                     const void* u, void* v, const int* len_out, const int* blk_off, const float* var, float* invstd) {
    const int vdt = ntype_of(d->io_dtype);
    if (ctx->gemm_mode == 0 && tc_fwd_supported(&ctx->tc, opdt, Cin, m.Cout, m.Tp))
        tc_gemm_fwd(&ctx->tc, L, opdt, w, u, nullptr, v, vdt, len_out, blk_off, m.B, Cin, m.Cout, m.Tp, nullptr, nullptr);
    else
        gemm_fwd_simt(L, opdt, w, u, nullptr, v, vdt, len_out, m.B, Cin, m.Cout, m.Tp);
    invstd_from_var(L, var, d->bn_eps, invstd, m.Cout);
}

Prologue length_prologue(const Dims& m, const int* len_in, int* len_out, int* nvalid, int* blk_off) {
    Prologue p;
    p.len_in = len_in; p.B = m.B; p.T_in = m.T; p.stride = m.s; p.len_out = len_out; p.nvalid = nvalid; p.blk_off = blk_off;
    return p;
}
bool needs_w16(const sc_block_desc* d, const Dims& m) { return op_dtype(d) != d->io_dtype && !m.full; }

int block_fwd_impl(sc_ctx* ctx, const Launch& L, const sc_block_desc* d, const Dims& m, BlockIO io,
                   const sc_block_params* p, sc_block_saved* sv, float* rmean, float* rvar,
                   const FwdScratch& f, const InferStats* inf = nullptr) {
    const int dt = d->io_dtype;
    if (!io.lengths_ready) {                                  // a later striding layer of an encoder
        Prologue pr = length_prologue(m, io.len_in, io.len_out, io.nvalid, io.blk_off);
        prologue(L, pr);
    }
    const int odt = op_dtype(d);
    // evaluation mode on whole rows: batch norm, residual and ReLU end the contraction, v is never stored
    const bool fused = inf && d->has_bn && !m.full && !io.phases && ctx->gemm_mode == 0 &&
                       tc_affine_supported(&ctx->tc, odt, m.B, m.Cin, m.Cout, m.Tp) &&
                       (d->residual != SC_RES_PROJ || tc_affine_supported(&ctx->tc, dt, m.B, m.Cres, m.Cout, m.Tp));
    ApplyArgs a{};
    a.v = sv->v; a.mean = inf ? inf->mean : sv->mean; a.invstd = sv->invstd; a.gamma = p->gamma; a.beta = p->beta;
    a.residual = d->residual; a.y = io.y; a.len_out = io.len_out;
    a.B = m.B; a.C = m.Cout; a.Tp = m.Tp; a.has_relu = d->has_relu; a.res_before_relu = d->res_before_relu;
    if (d->residual == SC_RES_IDENTITY) a.xres = io.xres;
    if (d->residual == SC_RES_PROJ) {
        a.vr = sv->vr; a.mean_r = inf ? inf->mean_r : sv->mean_r; a.invstd_r = sv->invstd_r; a.gamma_r = p->gamma_r; a.beta_r = p->beta_r;
    }
    if (io.phases) {
        a.phases = io.phases; a.B = m.B / io.phases; a.T = io.Td; a.len_out = io.len_dense;
        a.v_out = io.dense.v; a.vr_out = io.dense.vr; a.Cu = m.Cin;
    }
    StatsLayout left;              // statistics of the main branch that the apply step takes
    left.kind = -1;
    if (d->has_bn && d->residual == SC_RES_PROJ) {
        // the residual projection does not depend on the main branch: its contraction and statistics go to the
        // side stream and are joined just before the apply step
        fork_to_side(ctx, L, ctx->ev[4]);
        const Launch Ls = side_launch(ctx, L);
        const void* xr = io.xres;
        if (!io.res_clean) { mask_copy(Ls, dt, f.xr, io.xres, io.len_out, m.B, m.Cres, m.Tp); xr = f.xr; }
        if (fused) tc_gemm_affine(&ctx->tc, Ls, dt, p->wr, xr, sv->vr, SC_F16, AffineTail{inf->mean_r, inf->var_r, p->gamma_r, p->beta_r, d->bn_eps},
                                  io.len_out, io.blk_off, m.B, m.Cres, m.Cout, m.Tp);
        else if (inf) pointwise_fixed(ctx, Ls, d, m, m.Cres, dt, p->wr, xr, sv->vr, io.len_out, io.blk_off, inf->var_r, sv->invstd_r);
        else pointwise_bn(ctx, Ls, d, m, m.Cres, dt, p->wr, xr, sv->vr, io.len_out, io.nvalid, io.blk_off, sv->mean_r,
                          sv->invstd_r, f.partials_r, nullptr, nullptr);
        record_side(ctx, ctx->ev[5]);
    }
    if (m.full) {
        // block variant: one K-tap convolution over all input channels (it masks its input by len_in itself)
        const int vdt = d->has_bn ? ntype_of(dt) : dt;
        void* v = d->has_bn ? sv->v : io.y;
        const float* bias = !d->has_bn && d->has_bias ? p->bias : nullptr;
        const bool stats = d->has_bn && !inf;
        StatsLayout sl;
        if (ctx->gemm_mode == 0 && f.x_tm) {
            to_time_major(L, io.x, f.x_tm, io.len_in, m.B, m.Cin, m.T);
            split_taps(L, p->wp, f.taps, m.Cout, m.Cin, m.K, 0);
            tc_conv_fwd(&ctx->tc, L, dt, f.taps, f.x_tm, bias, v, vdt, io.len_out, io.blk_off, m.B, m.Cin, m.Cout, m.T, m.K, m.dil,
                        stats ? f.partials : nullptr, stats ? &sl : nullptr);
        } else {
            conv_fwd_simt(L, dt, p->wp, io.x, bias, v, vdt, io.len_in, io.len_out, m.B, m.Cin, m.Cout, m.T, m.Tp, m.K, m.s, m.dil);
        }
        if (!d->has_bn) return SC_OK;
        if (stats && apply_takes_stats(dt, a, sl)) left = sl;
        else if (stats) finalize_stats(L, d, m, sl, v, vdt, io.len_out, io.nvalid, io.blk_off, f.partials, sv->mean, sv->invstd, rmean, rvar);
        else invstd_from_var(L, inf->var, d->bn_eps, sv->invstd, m.Cout);
    }
    const void* u = nullptr;
    if (m.full) {
    } else if (d->has_dw) {
        if (ctx->gemm_mode == 0 && m.plain && dw_tma_supported(&ctx->tc, dt, m.B, m.T, m.K, m.s))
            dw_tma_fwd(&ctx->tc, L, dt, odt, io.x, p->wd, sv->u, io.len_in, io.len_out, m.B, m.Cin, m.T, m.K,
                       io.x_clean ? 1 : 0);
        else
            dw_fwd(L, dt, odt, io.x, p->wd, sv->u, io.len_in, io.len_out, m.B, m.Cin, m.T, m.Tp, m.K, m.s, m.dil);
        u = sv->u;
    } else if (io.x_clean) {
        u = io.x;
    } else {
        mask_copy(L, dt, sv->u, io.x, io.len_in, m.B, m.Cin, m.T);
        u = sv->u;
    }
    if (!d->has_bn) {   // linear layer: y = mask * (w u + bias), or its log-softmax over the channels
        // with the decoder tail the class scores stay in float32 until the log-softmax has been taken
        void* z = d->log_softmax ? (void*)f.zf32 : io.y;
        const int zdt = d->log_softmax ? (int)SC_F32 : dt;
        if (ctx->gemm_mode == 0 && tc_fwd_supported(&ctx->tc, dt, m.Cin, m.Cout, m.Tp)) {
            tc_gemm_fwd(&ctx->tc, L, dt, p->wp, u, d->has_bias ? p->bias : nullptr, z, zdt, io.len_out, io.blk_off, m.B,
                        m.Cin, m.Cout, m.Tp, nullptr, nullptr);
        } else {
            gemm_fwd_simt(L, dt, p->wp, u, d->has_bias ? p->bias : nullptr, z, zdt, io.len_out, m.B, m.Cin, m.Cout, m.Tp);
        }
        if (d->log_softmax) log_softmax_fwd(L, dt, f.zf32, io.y, io.len_out, m.B, m.Cout, m.Tp);
        return SC_OK;
    }
    const void* wp_op = p->wp;
    if (needs_w16(d, m)) wp_op = io.w16;
    if (fused) {
        AffineTail aff{inf->mean, inf->var, p->gamma, p->beta, d->bn_eps};
        aff.relu = d->has_relu; aff.res_before_relu = d->res_before_relu;
        if (d->residual == SC_RES_PROJ) { aff.add = sv->vr; aff.add_dtype = SC_F16; wait_side(ctx, L, ctx->ev[5]); }
        if (d->residual == SC_RES_IDENTITY) { aff.add = io.xres; aff.add_dtype = dt; }
        tc_gemm_affine(&ctx->tc, L, odt, wp_op, u, io.y, dt, aff, io.len_out, io.blk_off, m.B, m.Cin, m.Cout, m.Tp);
        return SC_OK;
    }
    if (m.full) {}
    else if (inf) pointwise_fixed(ctx, L, d, m, m.Cin, odt, wp_op, u, sv->v, io.len_out, io.blk_off, inf->var, sv->invstd);
    else pointwise_bn(ctx, L, d, m, m.Cin, odt, wp_op, u, sv->v, io.len_out, io.nvalid, io.blk_off, sv->mean, sv->invstd,
                      f.partials, rmean, rvar, &a, &left);
    if (d->residual == SC_RES_PROJ) wait_side(ctx, L, ctx->ev[5]);      // the projection branch (enqueued above on the side stream) is complete
    if (io.phases) { a.u = u; a.u_out = u ? io.dense.u : nullptr; }
    if (left.kind == 2)
        bn_apply_flat(L, dt, a, FlatStats{(const float4*)f.partials, left.grid, left.tiles_m, left.rows_per_tile, io.blk_off, io.nvalid,
                                          d->bn_eps, d->bn_momentum, sv->mean, sv->invstd, rmean, rvar});
    else if (left.kind == 0) bn_small_fwd(L, a, io.nvalid, d->bn_eps, d->bn_momentum, sv->mean, sv->invstd, rmean, rvar);
    else bn_apply(L, dt, a);
    return SC_OK;
}

// Operands of a packed forward pass.
struct FwdPack { void *x, *xres; int* len_dense; sc_block_saved sv; };
void plan_fwd_pack(const sc_block_desc* d, const Packed& k, Bump& ws, FwdPack* f) {
    const size_t e = esize(d->io_dtype), in = e * k.m.B * k.m.T;
    memset(f, 0, sizeof(*f));
    f->len_dense = (int*)ws.take(sizeof(int) * k.m.B / k.phases);
    f->x = ws.take(in * k.m.Cin);
    if (d->residual == SC_RES_PROJ) f->xres = ws.take(e * k.m.B * k.m.Cres * k.m.Tp);
    f->sv.u = ws.take(e * k.m.B * k.m.Cin * k.m.Tp);
    f->sv.v = ws.take((size_t)2 * k.m.B * k.m.Cout * k.m.Tp);
    if (d->residual == SC_RES_PROJ) f->sv.vr = ws.take((size_t)2 * k.m.B * k.m.Cout * k.m.Tp);
}
// The prologue of a single block's forward pass.
void enter(const Launch& L, const sc_block_desc* d, const Dims& m, const Packed& k, const FwdPack& fp, const FwdScratch& f,
           const sc_block_params* p, BlockIO& io, int* out_lengths) {
    Prologue pr = length_prologue(m, io.len_in, io.len_out, io.nvalid, io.blk_off);
    pr.len_user = out_lengths;
    if (k.phases > 1) { pr.phases = k.phases; pr.len_dense = fp.len_dense; }
    if (needs_w16(d, m)) { pr.convert(p->wp, f.w16, m.Cout * m.Cin); io.w16 = f.w16; }
    prologue(L, pr);
    io.lengths_ready = true;
}
// Packs the inputs and points io / sv (the caller's, dense) at the packed operands.
void enter_packed(const Launch& L, const sc_block_desc* d, const Dims& m, const Packed& k, const FwdPack& f, BlockIO& io,
                  sc_block_saved& sv) {
    PackList pl{};
    auto add = [&](const void* src, void* dst, int C, const int* len) { pl.src[pl.count] = src; pl.dst[pl.count] = dst; pl.C[pl.count] = C; pl.len[pl.count] = len; ++pl.count; };
    add(io.x, f.x, m.Cin, io.len_in);
    const bool own = d->residual == SC_RES_PROJ && io.xres == io.x && m.s == 1;       // the residual source is the input itself
    if (d->residual == SC_RES_PROJ && !own && m.s == 1) add(io.xres, f.xres, m.Cres, io.len_in);
    pack_frames(L, pl, m.B, m.T, k.Tq, k.phases);
    if (d->residual == SC_RES_PROJ && m.s != 1) {
        PackList pr{}; pr.count = 1; pr.src[0] = io.xres; pr.dst[0] = f.xres; pr.C[0] = m.Cres; pr.len[0] = io.len_out;
        pack_frames(L, pr, m.B, m.Tp, k.m.Tp, 1);
    }
    io.x = f.x;
    if (d->residual == SC_RES_PROJ) io.xres = own ? f.x : f.xres;
    io.x_clean = io.res_clean = true;
    io.phases = k.phases; io.Td = m.Tp; io.len_dense = k.phases > 1 ? f.len_dense : io.len_out;
    if (k.phases > 1) io.len_in = io.len_out;
    io.dense.u = sv.u; io.dense.v = sv.v; io.dense.vr = sv.vr;
    sv.u = f.sv.u; sv.v = f.sv.v; sv.vr = f.sv.vr;
}

// ---- backward scratch --------------------------------------------------------------------------
struct BwdScratch {
    int* len_out; int* nvalid; int* blk_off;
    float4 *partials, *coef, *coef_r;
    float *amax_part, *gmax;
    void *gv, *gvr, *gres, *gu, *gxr, *xr, *w16, *dz;
    void *x_tm, *gv_tm, *taps;           // operand copies of the non-separable convolution's tensor-core form
    void *gv16, *gvr16, *x16, *xr16;     // half copies for the weight gradients of bf16 layers (see block_bwd_impl)
    float* wpart; size_t wpart_bytes;
};

void plan_bwd(const sc_block_desc* d, const Dims& m, Bump& ws, BwdScratch* s, const TcState* tc) {
    const size_t e = esize(d->io_dtype);
    // gu holds the gradient w.r.t. the pointwise operand [B, C_in, T']; with the non-separable convolution it is the
    // staging tensor of the input gradient [B, C_in, T]
    const size_t act_out = e * m.B * m.Cout * m.Tp, act_in = e * m.B * m.Cin * (m.full ? m.T : m.Tp);
    s->len_out = (int*)ws.take(sizeof(int) * m.B);
    s->nvalid = (int*)ws.take(sizeof(int));
    s->blk_off = (int*)ws.take(sizeof(int) * (m.B + 1));
    s->partials = (float4*)ws.take(sizeof(float4) * m.B * m.Cout * bn_bwd_max_slots(m.Tp));
    s->coef = (float4*)ws.take(sizeof(float4) * m.Cout);
    s->coef_r = (float4*)ws.take(sizeof(float4) * m.Cout);
    s->amax_part = (float*)ws.take(sizeof(float) * m.B * m.Cout * bn_bwd_max_slots(m.Tp));
    s->gmax = (float*)ws.take(sizeof(float));
    s->w16 = (op_dtype(d) != d->io_dtype) ? ws.take((size_t)2 * m.Cout * m.Cin) : nullptr;
    s->gv = ws.take(act_out);
    s->dz = d->log_softmax ? ws.take(act_out) : nullptr;
    s->gvr = d->residual == SC_RES_PROJ ? ws.take(act_out) : nullptr;
    s->gres = d->residual == SC_RES_IDENTITY ? ws.take(act_out) : nullptr;
    s->gu = ws.take(act_in);
    s->gxr = d->residual == SC_RES_PROJ ? ws.take(e * m.B * m.Cres * m.Tp) : nullptr;
    s->xr = d->residual == SC_RES_PROJ ? ws.take(e * m.B * m.Cres * m.Tp) : nullptr;
    const bool bf = d->io_dtype == SC_BF16 && d->has_bn && !m.full;
    s->gv16 = (bf && !d->has_dw) ? ws.take(act_out) : nullptr;
    s->x16 = (bf && !d->has_dw) ? ws.take(act_in) : nullptr;
    s->gvr16 = (bf && d->residual == SC_RES_PROJ) ? ws.take(act_out) : nullptr;
    s->xr16 = (bf && d->residual == SC_RES_PROJ) ? ws.take(e * m.B * m.Cres * m.Tp) : nullptr;
    size_t wb = gemm_wgrad_simt_scratch_bytes(m.B, std::max(m.Cin, m.Cres), m.Cout);
    wb = std::max(wb, tc_wgrad_scratch_bytes(tc, std::max(m.Cin, m.Cres), m.Cout));
    wb = std::max(wb, dw_wgrad_scratch_bytes(m.B, m.Cin, m.K));
    if (m.full) wb = std::max(wb, conv_wgrad_scratch_bytes(m.B, m.Cin, m.Cout, m.K));
    const bool conv = conv_on_tc(tc, d, m);
    if (conv) wb = std::max(wb, tc_conv_wgrad_scratch_bytes(m.B, m.Cin, m.Cout, m.T, m.K));
    s->x_tm = conv ? ws.take((size_t)2 * m.B * m.Cin * m.T) : nullptr;
    s->gv_tm = conv ? ws.take((size_t)2 * m.B * m.Cout * m.T) : nullptr;
    s->taps = conv ? ws.take((size_t)2 * m.Cin * m.Cout * m.K) : nullptr;
    s->wpart = (float*)ws.take(wb);
    s->wpart_bytes = wb;
}

void pointwise_wgrad(sc_ctx* ctx, const Launch& L, int dt, const void* gv, const void* u, float* dw,
                     float* part, int acc, int B, int Cin, int Cout, int Tp, const int* len_out,
                     const float* gmax) {
    if (ctx->gemm_mode == 0 && tc_wgrad_supported(&ctx->tc, dt, Cin, Cout, Tp))
        tc_gemm_wgrad(&ctx->tc, L, dt, gv, u, dw, part, acc, B, Cin, Cout, Tp, len_out, gmax);
    else
        gemm_wgrad_simt(L, dt, gv, u, dw, part, acc, B, Cin, Cout, Tp, gmax);
}
void pointwise_dgrad(sc_ctx* ctx, const Launch& L, int dt, const void* w, const void* gv, void* gu, int B,
                     int Cin, int Cout, int Tp, const int* len_out, const int* blk_off) {
    if (ctx->gemm_mode == 0 && tc_dgrad_supported(&ctx->tc, dt, Cin, Cout, Tp))
        tc_gemm_dgrad(&ctx->tc, L, dt, w, gv, gu, B, Cin, Cout, Tp, len_out, blk_off);
    else
        gemm_dgrad_simt(L, dt, w, gv, gu, B, Cin, Cout, Tp);
}

struct BwdIO {
    const void *dy, *x, *xres, *y;
    void *dx, *dx_res; const void* dx_add;
    const int* len_in; const int* len_out; const int* nvalid; const int* blk_off;
    bool x_clean, res_clean;
    const void* w16;             // float16 copy of wp (see BlockIO)
    bool fork_early;             // a single block: nothing follows that the weight gradients could overlap
    cudaEvent_t done;            // recorded on the side stream after this layer's last side-stream kernel
    int phases, Td; uint32_t total_dense;      // packed block: dy, y and the saved v, vr are dense [., ., Td]; the rest is packed
    float* gmax;                 // where the bound on |gv| collects; already zero
};

int block_bwd_impl(sc_ctx* ctx, const Launch& L, const sc_block_desc* d, const Dims& m, BwdIO io,
                   const sc_block_params* p, const sc_block_saved* sv, sc_block_grads* g, int acc,
                   const BwdScratch& s) {
    const int dt = d->io_dtype;
    const int odt = op_dtype(d);
    // gv (and gu after it) is kept scaled by a power of two whenever it is a library-internal 16-bit
    // tensor, so that neither a tiny nor a huge upstream gradient leaves the half range
    // bf16 layers whose gv / gvr stay in bf16 (no depthwise step; the residual projection) get a scaled
    // half copy of that gradient, and of the other operand, for their weight-gradient contraction: with
    // 8 significand bits the rounding of the gradient alone uses most of the error budget of dwp / dwr
    const bool tc_ok = ctx->gemm_mode == 0;
    const bool half_gv = dt == SC_BF16 && d->has_bn && !d->has_dw && !m.full && s.gv16 && tc_ok &&
                         tc_wgrad_supported(&ctx->tc, SC_F16, m.Cin, m.Cout, m.Tp);
    const bool half_gvr = dt == SC_BF16 && d->has_bn && d->residual == SC_RES_PROJ && s.gvr16 && tc_ok &&
                          tc_wgrad_supported(&ctx->tc, SC_F16, m.Cres, m.Cout, m.Tp);
    float* gmax = (dt != SC_F32 && d->has_bn && (d->has_dw || half_gv || half_gvr)) ? io.gmax : nullptr;
    const void* dy = io.dy;
    if (d->log_softmax) {      // upstream gradient is w.r.t. the log-probabilities: back through the log-softmax first
        log_softmax_bwd(L, dt, s.dz, io.dy, io.y, io.len_out, m.B, m.Cout, m.Tp);
        dy = s.dz;
    }
    BnBwdArgs a{};
    a.amax_part = s.amax_part; a.gmax = gmax; a.gv_dtype = odt;
    a.gv_scaled = (gmax && d->has_dw) ? 1 : 0;
    a.gv16 = half_gv ? s.gv16 : nullptr; a.gvr16 = half_gvr ? s.gvr16 : nullptr;
    a.g = dy; a.y = io.y; a.v = sv->v; a.vr = sv->vr;
    a.mean = sv->mean; a.mean_r = sv->mean_r; a.invstd = sv->invstd; a.invstd_r = sv->invstd_r; a.gamma = p->gamma; a.beta = p->beta;
    a.len_out = io.len_out; a.nvalid = io.nvalid;
    a.B = m.B; a.C = m.Cout; a.Tp = m.Tp; a.has_bn = d->has_bn; a.has_relu = d->has_relu;
    a.res_before_relu = d->res_before_relu; a.residual = d->residual;
    a.partials = s.partials; a.coef = s.coef; a.coef_r = s.coef_r;
    a.gv = s.gv; a.gvr = s.gvr;
    // identity residual: its gradient is the gated upstream gradient itself
    a.gres = (d->residual == SC_RES_IDENTITY) ? (io.dx_res ? io.dx_res : s.gres) : nullptr;
    a.phases = io.phases; a.T = io.Td; a.total_dense = io.total_dense;
    a.skip_padding = tc_ok && !m.full && tc_bwd_blockwise(&ctx->tc, odt, m.B, m.Cin, m.Cout, m.Tp) &&
                     (d->residual != SC_RES_PROJ || tc_bwd_blockwise(&ctx->tc, dt, m.B, m.Cres, m.Cout, m.Tp));
    bn_bwd(L, dt, a, p->gamma, p->gamma_r, g->dgamma, g->dbeta, g->dgamma_r, g->dbeta_r, d->has_bias ? g->dbias : nullptr, acc);
    const bool conv_tc = tc_ok && conv_on_tc(&ctx->tc, d, m);
    if (conv_tc) to_time_major(L, s.gv, s.gv_tm, io.len_out, m.B, m.Cout, m.T);

    // The weight gradients are off the critical path (nothing later in the backward pass reads them): they run on the
    // side stream.  They are enqueued after the input-gradient kernels of this stream: the host issues launches in
    // program order, and kernels of the critical path that sit behind side-stream launches in that order start late
    // whenever the GPU is ahead of the host.  One event, recorded behind this layer's last main-stream kernel, releases
    // them (an event between two kernels ends the programmatic overlap of that pair, so there is only one per layer);
    // they then overlap the next layer's main-stream kernels.  A block call has no next layer: there they are released as
    // soon as their operands are complete and overlap this block's own input-gradient kernels.
    const Launch Ls = side_launch(ctx, L);
    auto pointwise_weight_gradients = [&]() {
        const void* u = d->has_dw ? sv->u : (io.x_clean ? io.x : sv->u);
        if (conv_tc) {
            to_time_major(Ls, io.x, s.x_tm, io.len_in, m.B, m.Cin, m.T);
            tc_conv_wgrad(&ctx->tc, Ls, dt, s.gv_tm, s.x_tm, g->dwp, s.wpart, acc, io.len_out, m.B, m.Cin, m.Cout, m.T, m.K, m.dil);
        } else if (m.full) {
            conv_wgrad_simt(Ls, dt, s.gv, io.x, g->dwp, s.wpart, acc, io.len_in, io.len_out, m.B, m.Cin, m.Cout, m.T, m.Tp, m.K, m.s, m.dil);
        } else if (half_gv) {
            mask_convert_f16(Ls, s.x16, io.x, io.len_in, m.B, m.Cin, m.T);
            pointwise_wgrad(ctx, Ls, SC_F16, s.gv16, s.x16, g->dwp, s.wpart, acc, m.B, m.Cin, m.Cout, m.Tp, io.len_out, gmax);
        } else {
            pointwise_wgrad(ctx, Ls, odt, s.gv, u, g->dwp, s.wpart, acc, m.B, m.Cin, m.Cout, m.Tp, io.len_out,
                            a.gv_scaled ? gmax : nullptr);
        }
        if (d->residual == SC_RES_PROJ) {
            if (half_gvr) {
                mask_convert_f16(Ls, s.xr16, io.xres, io.len_out, m.B, m.Cres, m.Tp);
                pointwise_wgrad(ctx, Ls, SC_F16, s.gvr16, s.xr16, g->dwr, s.wpart, acc, m.B, m.Cres, m.Cout, m.Tp, io.len_out, gmax);
            } else {
                const void* xr = io.xres;
                if (!io.res_clean) { mask_copy(Ls, dt, s.xr, io.xres, io.len_out, m.B, m.Cres, m.Tp); xr = s.xr; }
                pointwise_wgrad(ctx, Ls, dt, s.gvr, xr, g->dwr, s.wpart, acc, m.B, m.Cres, m.Cout, m.Tp, io.len_out, nullptr);
            }
        }
    };
    auto tap_gradients = [&]() {
        if (d->has_dw && !m.full) {
            if (ctx->gemm_mode == 0 && m.plain && dw_wgrad_tc_supported(&ctx->tc, dt, m.B, m.T, m.K, m.s))
                dw_wgrad_tc(&ctx->tc, Ls, dt, odt, s.gu, io.x, g->dwd, s.wpart, acc, gmax, io.len_in, io.len_out, m.B, m.Cin,
                            m.T, m.K, io.x_clean ? 1 : 0);
            else
                dw_wgrad(Ls, dt, odt, s.gu, io.x, g->dwd, s.wpart, acc, gmax, io.len_in, io.len_out, m.B, m.Cin, m.T, m.Tp, m.K, m.s, m.dil);
        }
    };

    if (io.fork_early) {
        fork_to_side(ctx, L, ctx->ev[0]);               // gv, gvr and the half copies are complete
        pointwise_weight_gradients();
    }
    const void* wp_op = p->wp;
    if (needs_w16(d, m)) wp_op = io.w16;
    const void* extra = nullptr;    // residual-path gradient to fold into dx
    if (d->residual == SC_RES_PROJ) {
        void* tgt = io.dx_res ? io.dx_res : s.gxr;
        if (io.dx_res || io.dx) pointwise_dgrad(ctx, L, dt, p->wr, s.gvr, tgt, m.B, m.Cres, m.Cout, m.Tp, io.len_out, io.blk_off);
        if (!io.dx_res) extra = s.gxr;
    } else if (d->residual == SC_RES_IDENTITY && !io.dx_res) {
        extra = s.gres;
    }

    if (m.full) {
        if (io.dx) {
            void* tgt = (!io.dx_add && !extra) ? io.dx : s.gu;
            if (conv_tc) {
                split_taps(L, p->wp, s.taps, m.Cout, m.Cin, m.K, 1);
                tc_conv_dgrad(&ctx->tc, L, dt, s.taps, s.gv_tm, tgt, io.len_in, io.blk_off, m.B, m.Cin, m.Cout, m.T, m.K, m.dil);
            } else {
                conv_dgrad_simt(L, dt, p->wp, s.gv, tgt, io.len_in, io.len_out, m.B, m.Cin, m.Cout, m.T, m.Tp, m.K, m.s, m.dil);
            }
            if (tgt != io.dx) ew_add_masked(L, dt, io.dx, s.gu, io.dx_add, extra, io.len_in, m.B, m.Cin, m.T);
        }
    } else if (d->has_dw) {
        pointwise_dgrad(ctx, L, odt, wp_op, s.gv, s.gu, m.B, m.Cin, m.Cout, m.Tp, io.len_out, io.blk_off);
        if (io.fork_early) {
            fork_to_side(ctx, L, ctx->ev[1]);           // gu is complete
            tap_gradients();
        }
        if (io.dx) {
            if (ctx->gemm_mode == 0 && m.plain && dw_tma_supported(&ctx->tc, dt, m.B, m.T, m.K, m.s))
                dw_tma_dgrad(&ctx->tc, L, dt, odt, s.gu, p->wd, io.dx, io.dx_add, extra, gmax, io.len_in, io.len_out, m.B,
                             m.Cin, m.T, m.K);
            else
                dw_dgrad(L, dt, odt, s.gu, p->wd, io.dx, io.dx_add, extra, gmax, io.len_in, io.len_out, m.B, m.Cin, m.T,
                         m.Tp, m.K, m.s, m.dil);
        }
    } else if (io.dx) {
        if (!io.dx_add && !extra) {
            pointwise_dgrad(ctx, L, dt, p->wp, s.gv, io.dx, m.B, m.Cin, m.Cout, m.Tp, io.len_out, io.blk_off);
        } else {
            pointwise_dgrad(ctx, L, dt, p->wp, s.gv, s.gu, m.B, m.Cin, m.Cout, m.Tp, io.len_out, io.blk_off);
            ew_add_masked(L, dt, io.dx, s.gu, io.dx_add, extra, io.len_in, m.B, m.Cin, m.T);
        }
    }
    if (!io.fork_early) {
        fork_to_side(ctx, L, ctx->ev[0]);               // gv, gvr, gu and the half copies are complete
        pointwise_weight_gradients();
        tap_gradients();
    }
    // the caller joins: it waits for io.done on its stream before it reuses this scratch or returns
    if (io.done) record_side(ctx, io.done);
    return SC_OK;
}

// Packed operands of a backward pass.
struct BwdPack { void *x, *xres, *u, *dx, *dx_res, *dx_add; int* len_dense; };
void plan_bwd_pack(const sc_block_desc* d, const Packed& k, Bump& ws, BwdPack* b) {
    const size_t e = esize(d->io_dtype), in = e * k.m.B * k.m.Cin * k.m.T;
    memset(b, 0, sizeof(*b));
    b->len_dense = (int*)ws.take(sizeof(int) * k.m.B / k.phases);
    b->x = ws.take(in); b->dx = ws.take(in); b->dx_add = ws.take(in);
    b->u = ws.take(e * k.m.B * k.m.Cin * k.m.Tp);
    if (d->residual != SC_RES_NONE) { b->xres = ws.take(e * k.m.B * k.m.Cres * k.m.Tp); b->dx_res = ws.take(e * k.m.B * k.m.Cres * k.m.Tp); }
}

int check_params(const sc_block_desc* d, const sc_block_params* p) {
    if (!p || !p->wp) return SC_ERR_NULL;
    if (d->has_dw && !p->wd) return SC_ERR_NULL;
    if (d->has_bn && (!p->gamma || !p->beta)) return SC_ERR_NULL;
    if (d->has_bias && !p->bias) return SC_ERR_NULL;
    if (d->residual == SC_RES_PROJ && (!p->wr || !p->gamma_r || !p->beta_r)) return SC_ERR_NULL;
    return SC_OK;
}
int check_saved(const sc_block_desc* d, const sc_block_saved* s, bool x_clean) {
    if (!s) return SC_ERR_NULL;
    if (!d->full_conv && (d->has_dw || !x_clean) && !s->u) return SC_ERR_NULL;
    if (d->has_bn && (!s->v || !s->mean || !s->invstd)) return SC_ERR_NULL;
    if (d->residual == SC_RES_PROJ && (!s->vr || !s->mean_r || !s->invstd_r)) return SC_ERR_NULL;
    return SC_OK;
}
int check_grads(const sc_block_desc* d, const sc_block_grads* g) {
    if (!g || !g->dwp) return SC_ERR_NULL;
    if (d->has_dw && !g->dwd) return SC_ERR_NULL;
    if (d->has_bn && (!g->dgamma || !g->dbeta)) return SC_ERR_NULL;
    if (d->has_bias && !g->dbias) return SC_ERR_NULL;
    if (d->residual == SC_RES_PROJ && (!g->dwr || !g->dgamma_r || !g->dbeta_r)) return SC_ERR_NULL;
    return SC_OK;
}

int finish(sc_ctx* ctx) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { fprintf(stderr, "sepconv: CUDA error: %s\n", cudaGetErrorString(e)); return SC_ERR_CUDA; }
    (void)ctx;
    return SC_OK;
}

// ---- calls through the graph cache -----------------------------------------------------------------
enum CallTag : uint32_t { CALL_FWD = 1, CALL_BWD, CALL_INFER, CALL_ENC, CALL_ENC_INFER };
void key_tensor(CallKey& k, const sc_tensor* t) { k.add(t, offsetof(sc_tensor, tag) + sizeof(t->tag)); }
void key_begin(sc_ctx* ctx, CallTag tag, void* ws, size_t ws_bytes) {
    CallKey& k = ctx->key;
    k.reset(tag);
    k.val(ws); k.val(ws_bytes);
    k.val(ctx->gemm_mode); k.val(ctx->overlap); k.val(ctx->pdl); k.val(ctx->tc.flat_shape);
}
// The key holds every argument, so a replayed call is one that has passed validation before.  Calls that are being
// timed launch by launch are never replayed.
template <typename F> int run_call(sc_ctx* ctx, void* stream, F&& body) {
    auto go = [&](cudaStream_t s) -> int {
        return body(Launch{s, ctx->status_dev, &ctx->launches, &ctx->prof, ctx->gemm_mode, ctx->pdl, ctx->fresh});
    };
    if (ctx->prof.filter != -2) return go((cudaStream_t)stream);
    return ctx->graphs.run(ctx->key, (cudaStream_t)stream, &ctx->launches, SC_ERR_CUDA, go);
}

#define SC_TRY(expr) do { int _r = (expr); if (_r != SC_OK) return _r; } while (0)

}  // namespace

// =================================================================================================
extern "C" {

int sepconv_ctx_create(sc_ctx** out, int device) {
    if (!out) return SC_ERR_NULL;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) return SC_ERR_CUDA;
    if (prop.major != 10) return SC_ERR_ARCH;
    if (cudaSetDevice(device) != cudaSuccess) return SC_ERR_CUDA;
    sc_ctx* c = new (std::nothrow) sc_ctx();
    if (!c) return SC_ERR_CUDA;
    c->device = device;
    c->sm_count = prop.multiProcessorCount;
    if (cudaMalloc(&c->status_dev, 64) != cudaSuccess) { delete c; return SC_ERR_CUDA; }
    cudaMemset(c->status_dev, 0, 64);
    int r = tc_init(&c->tc, device, c->sm_count);
    if (r != SC_OK) { cudaFree(c->status_dev); delete c; return r; }
    bool ok = cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) == cudaSuccess;
    for (int i = 0; i < 8 && ok; ++i) ok = cudaEventCreateWithFlags(&c->ev[i], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) { sepconv_ctx_destroy(c); return SC_ERR_CUDA; }
    *out = c;
    return SC_OK;
}

void sepconv_ctx_destroy(sc_ctx* ctx) {
    if (!ctx) return;
    ctx->graphs.clear();
    for (cudaEvent_t e : ctx->prof.events) cudaEventDestroy(e);
    for (cudaEvent_t e : ctx->ev) if (e) cudaEventDestroy(e);
    if (ctx->side) cudaStreamDestroy(ctx->side);
    cudaFree(ctx->status_dev);
    tc_destroy(&ctx->tc);
    delete ctx;
}

int sepconv_last_status(sc_ctx* ctx, void* stream) {
    if (!ctx) return SC_ERR_NULL;
    int h = 0;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemcpyAsync(&h, ctx->status_dev, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return SC_ERR_CUDA;
    if (cudaMemsetAsync(ctx->status_dev, 0, sizeof(int), st) != cudaSuccess) return SC_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SC_ERR_CUDA;
    return h;
}

const char* sepconv_strerror(int s) {
    switch (s) {
        case SC_OK: return "ok";
        case SC_ERR_NULL: return "a required pointer is null";
        case SC_ERR_INCOMPATIBLE: return "incompatible tensor type (dtype, rank or axis tags)";
        case SC_ERR_DIM_INCOMPATIBLE: return "an axis size disagrees with the descriptor";
        case SC_ERR_TRANSPOSED: return "axes are transposed or the tensor is not dense [batch, channel, time]";
        case SC_ERR_ALIGNMENT: return "pointer is not 16-byte aligned";
        case SC_ERR_UNSUPPORTED: return "unsupported block configuration";
        case SC_ERR_WORKSPACE: return "workspace is null or too small";
        case SC_ERR_LENGTHS: return "a length lies outside [1, T]";
        case SC_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait ran out";
        case SC_ERR_ARCH: return "device is not compute capability 10.x";
        case SC_ERR_CUDA: return "a CUDA call failed";
        case SC_ERR_RANGE: return "an intermediate value left the float16 range and was clamped";
        default: return "unknown status";
    }
}

int sepconv_selftest_bounded_wait(sc_ctx* ctx, void* cuda_stream) {
    if (!ctx) return SC_ERR_NULL;
    Launch L{(cudaStream_t)cuda_stream, ctx->status_dev, &ctx->launches, &ctx->prof, ctx->gemm_mode, ctx->pdl};
    selftest_bounded_wait(L);
    return finish(ctx);
}

int sepconv_set_tile_shape(sc_ctx* ctx, int shape) {
    if (!ctx) return SC_ERR_NULL;
    if (shape < 0 || shape > 5) return SC_ERR_UNSUPPORTED;
    ctx->tc.flat_shape = shape;
    return SC_OK;
}

int sepconv_set_overlap(sc_ctx* ctx, int on) {
    if (!ctx) return SC_ERR_NULL;
    if (on < 0 || on > 3) return SC_ERR_UNSUPPORTED;
    ctx->overlap = on & 1;
    ctx->pdl = (on >> 1) & 1;
    return SC_OK;
}

int sepconv_set_gemm_mode(sc_ctx* ctx, int mode) {
    if (!ctx) return SC_ERR_NULL;
    if (mode != 0 && mode != 1) return SC_ERR_UNSUPPORTED;
    ctx->gemm_mode = mode;
    return SC_OK;
}

int64_t sepconv_launch_count(sc_ctx* ctx) { return ctx ? ctx->launches : 0; }

int sepconv_profile_begin(sc_ctx* ctx, int kernel_class, int max_launches) {
    if (!ctx) return SC_ERR_NULL;
    if (kernel_class < -1 || kernel_class >= KC_COUNT || max_launches < 1) return SC_ERR_UNSUPPORTED;
    Prof& p = ctx->prof;
    while (p.events.size() < (size_t)2 * max_launches) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return SC_ERR_CUDA;
        p.events.push_back(e);
    }
    p.recs.clear(); p.used = 0; p.filter = kernel_class;
    return SC_OK;
}

int sepconv_profile_end(sc_ctx* ctx, void* cuda_stream, double* ms, int64_t* launches, double* bytes,
                        double* flops) {
    if (!ctx || !ms || !launches || !bytes || !flops) return SC_ERR_NULL;
    Prof& p = ctx->prof;
    p.filter = -2;
    if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess) return SC_ERR_CUDA;
    for (int c = 0; c < KC_COUNT; ++c) { ms[c] = 0; launches[c] = 0; bytes[c] = 0; flops[c] = 0; }
    for (const Prof::Rec& r : p.recs) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, p.events[r.e0], p.events[r.e0 + 1]) != cudaSuccess) return SC_ERR_CUDA;
        ms[r.cls] += t; launches[r.cls] += 1; bytes[r.cls] += r.bytes; flops[r.cls] += r.flops;
    }
    p.recs.clear(); p.used = 0;
    return SC_OK;
}

int sepconv_kernel_class_count(void) { return KC_COUNT; }
const char* sepconv_kernel_class_name(int c) { return kclass_name(c); }

int sepconv_workspace_bytes(const sc_block_desc* desc, size_t* fwd, size_t* bwd) {
    Dims m;
    SC_TRY(desc_dims(desc, &m));
    const Packed k = plan_packed(desc, m);
    if (fwd) {
        Bump b(nullptr, 0); FwdScratch f; plan_fwd(desc, m, b, &f, nullptr); *fwd = b.off + 256;
        if (k.phases) { Bump q(nullptr, 0); FwdPack fp; plan_fwd(desc, k.m, q, &f, nullptr); plan_fwd_pack(desc, k, q, &fp); *fwd = std::max(*fwd, q.off + 256); }
    }
    if (bwd) {
        Bump b(nullptr, 0); BwdScratch s; plan_bwd(desc, m, b, &s, nullptr); *bwd = b.off + 256;
        if (k.phases) { Bump q(nullptr, 0); BwdPack bp; plan_bwd(desc, k.m, q, &s, nullptr); plan_bwd_pack(desc, k, q, &bp); *bwd = std::max(*bwd, q.off + 256); }
    }
    return SC_OK;
}

namespace {
int fwd_call(sc_ctx* ctx, const Launch& L, const sc_block_desc* desc, const sc_tensor* x, const sc_tensor* x_res,
             const int32_t* lengths_dev, const sc_block_params* params, sc_tensor* y, int32_t* out_lengths_dev,
             sc_block_saved* saved, float* running_mean, float* running_var, void* workspace, size_t workspace_bytes,
             bool dense_if_short) {
    Dims m;
    SC_TRY(desc_dims(desc, &m));
    const int dt = desc->io_dtype;
    SC_TRY(check_tensor(x, dt, m.B, m.Cin, m.T));
    SC_TRY(check_tensor(y, dt, m.B, m.Cout, m.Tp));
    if (desc->residual != SC_RES_NONE) {
        if (x_res) SC_TRY(check_tensor(x_res, dt, m.B, m.Cres, m.Tp));
        else if (m.s != 1 || m.Cres != m.Cin) return SC_ERR_UNSUPPORTED;
    }
    SC_TRY(check_params(desc, params));
    SC_TRY(check_saved(desc, saved, false));
    if (!workspace) return SC_ERR_WORKSPACE;
    Packed pk;
    if (ctx->gemm_mode == 0) pk = plan_packed(desc, m);
    FwdScratch f; FwdPack fp;
    Bump ws(workspace, workspace_bytes);
    plan_fwd(desc, pk.phases ? pk.m : m, ws, &f, &ctx->tc);
    if (pk.phases) plan_fwd_pack(desc, pk, ws, &fp);
    if (!ws.ok() && dense_if_short) {
        pk = Packed();
        ws = Bump(workspace, workspace_bytes);
        plan_fwd(desc, m, ws, &f, &ctx->tc, false);
    }
    if (!ws.ok()) return SC_ERR_WORKSPACE;
    BlockIO io{};
    io.x = x->ptr; io.xres = desc->residual != SC_RES_NONE ? (x_res ? x_res->ptr : x->ptr) : nullptr;
    io.y = y->ptr; io.len_in = lengths_dev; io.len_out = f.len_out; io.nvalid = f.nvalid; io.blk_off = f.blk_off;
    io.x_clean = false; io.res_clean = false; io.lengths_ready = false;
    sc_block_saved sv = *saved;
    enter(L, desc, m, pk, fp, f, params, io, out_lengths_dev);
    if (pk.phases) enter_packed(L, desc, m, pk, fp, io, sv);
    SC_TRY(block_fwd_impl(ctx, L, desc, pk.phases ? pk.m : m, io, params, &sv, running_mean, running_var, f));
    return finish(ctx);
}
}  // namespace

int sepconv_fwd(sc_ctx* ctx, const sc_block_desc* desc, const sc_tensor* x, const sc_tensor* x_res,
                const int32_t* lengths_dev, const sc_block_params* params, sc_tensor* y,
                int32_t* out_lengths_dev, sc_block_saved* saved, float* running_mean, float* running_var,
                void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!ctx || !lengths_dev || !desc) return SC_ERR_NULL;
    CallKey& k = ctx->key;
    key_begin(ctx, CALL_FWD, workspace, workspace_bytes);
    k.add(desc, sizeof(*desc)); key_tensor(k, x); key_tensor(k, x_res); k.val(lengths_dev); k.add(params, sizeof(*params));
    key_tensor(k, y); k.val(out_lengths_dev); k.add(saved, sizeof(*saved)); k.val(running_mean); k.val(running_var);
    return run_call(ctx, cuda_stream, [&](const Launch& L) {
        return fwd_call(ctx, L, desc, x, x_res, lengths_dev, params, y, out_lengths_dev, saved, running_mean, running_var, workspace,
                        workspace_bytes, false);
    });
}

namespace {
// scratch of the evaluation-mode forward: the training forward's scratch plus the tensors that call would save
struct InferScratch { FwdScratch f; sc_block_saved sv; };
void plan_infer(const sc_block_desc* d, const Dims& m, Bump& ws, InferScratch* q, const TcState* tc) {
    plan_fwd(d, m, ws, &q->f, tc);
    memset(&q->sv, 0, sizeof(q->sv));
    const size_t e = esize(d->io_dtype), en = dtype_size(ntype_of(d->io_dtype));
    q->sv.u = ws.take(e * m.B * m.Cin * m.Tp);
    if (d->has_bn) { q->sv.v = ws.take(en * m.B * m.Cout * m.Tp); q->sv.invstd = (float*)ws.take(4 * m.Cout); }
    if (d->residual == SC_RES_PROJ) { q->sv.vr = ws.take(en * m.B * m.Cout * m.Tp); q->sv.invstd_r = (float*)ws.take(4 * m.Cout); }
}
}  // namespace

int sepconv_infer_workspace_bytes(const sc_block_desc* desc, size_t* bytes) {
    if (!bytes) return SC_ERR_NULL;
    Dims m;
    SC_TRY(desc_dims(desc, &m));
    Bump b(nullptr, 0); InferScratch q; plan_infer(desc, m, b, &q, nullptr);
    *bytes = b.off + 256;
    const Packed k = plan_packed(desc, m);
    if (k.phases) {
        Bump c(nullptr, 0); FwdPack fp; plan_infer(desc, k.m, c, &q, nullptr); plan_fwd_pack(desc, k, c, &fp);
        *bytes = std::max(*bytes, c.off + 256);
    }
    return SC_OK;
}

namespace {
int infer_call(sc_ctx* ctx, const Launch& L, const sc_block_desc* desc, const sc_tensor* x, const sc_tensor* x_res,
               const int32_t* lengths_dev, const sc_block_params* params, const float* running_mean,
               const float* running_var, const float* running_mean_r, const float* running_var_r, sc_tensor* y,
               int32_t* out_lengths_dev, void* workspace, size_t workspace_bytes) {
    Dims m;
    SC_TRY(desc_dims(desc, &m));
    const int dt = desc->io_dtype;
    SC_TRY(check_tensor(x, dt, m.B, m.Cin, m.T));
    SC_TRY(check_tensor(y, dt, m.B, m.Cout, m.Tp));
    if (desc->residual != SC_RES_NONE) {
        if (x_res) SC_TRY(check_tensor(x_res, dt, m.B, m.Cres, m.Tp));
        else if (m.s != 1 || m.Cres != m.Cin) return SC_ERR_UNSUPPORTED;
    }
    SC_TRY(check_params(desc, params));
    if (desc->has_bn && (!running_mean || !running_var)) return SC_ERR_NULL;
    if (desc->residual == SC_RES_PROJ && (!running_mean_r || !running_var_r)) return SC_ERR_NULL;
    if (!workspace) return SC_ERR_WORKSPACE;
    Packed pk;
    if (ctx->gemm_mode == 0) pk = plan_packed(desc, m);
    Bump ws(workspace, workspace_bytes);
    InferScratch q; FwdPack fp;
    plan_infer(desc, pk.phases ? pk.m : m, ws, &q, &ctx->tc);
    if (pk.phases) plan_fwd_pack(desc, pk, ws, &fp);
    if (!ws.ok()) return SC_ERR_WORKSPACE;
    BlockIO io{};
    io.x = x->ptr; io.xres = desc->residual != SC_RES_NONE ? (x_res ? x_res->ptr : x->ptr) : nullptr;
    io.y = y->ptr; io.len_in = lengths_dev; io.len_out = q.f.len_out; io.nvalid = q.f.nvalid; io.blk_off = q.f.blk_off;
    InferStats inf{running_mean, running_var, running_mean_r, running_var_r};
    enter(L, desc, m, pk, fp, q.f, params, io, out_lengths_dev);
    if (pk.phases) { enter_packed(L, desc, m, pk, fp, io, q.sv); memset(&io.dense, 0, sizeof(io.dense)); }
    SC_TRY(block_fwd_impl(ctx, L, desc, pk.phases ? pk.m : m, io, params, &q.sv, nullptr, nullptr, q.f, &inf));
    return finish(ctx);
}
}  // namespace

int sepconv_infer(sc_ctx* ctx, const sc_block_desc* desc, const sc_tensor* x, const sc_tensor* x_res,
                  const int32_t* lengths_dev, const sc_block_params* params, const float* running_mean,
                  const float* running_var, const float* running_mean_r, const float* running_var_r, sc_tensor* y,
                  int32_t* out_lengths_dev, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!ctx || !lengths_dev || !desc) return SC_ERR_NULL;
    CallKey& k = ctx->key;
    key_begin(ctx, CALL_INFER, workspace, workspace_bytes);
    k.add(desc, sizeof(*desc)); key_tensor(k, x); key_tensor(k, x_res); k.val(lengths_dev); k.add(params, sizeof(*params));
    k.val(running_mean); k.val(running_var); k.val(running_mean_r); k.val(running_var_r);
    key_tensor(k, y); k.val(out_lengths_dev);
    return run_call(ctx, cuda_stream, [&](const Launch& L) { return infer_call(ctx, L, desc, x, x_res, lengths_dev, params, running_mean, running_var, running_mean_r,
                          running_var_r, y, out_lengths_dev, workspace, workspace_bytes); });
}

namespace {
int bwd_call(sc_ctx* ctx, const Launch& L, const sc_block_desc* desc, const sc_tensor* dy, const sc_tensor* x, const sc_tensor* x_res,
             const sc_tensor* y, const int32_t* lengths_dev, const sc_block_params* params, const sc_block_saved* saved,
             sc_tensor* dx, sc_tensor* dx_res, const sc_tensor* dx_add, sc_block_grads* grads, int accumulate,
             void* workspace, size_t workspace_bytes) {
    Dims m;
    SC_TRY(desc_dims(desc, &m));
    const int dt = desc->io_dtype;
    SC_TRY(check_tensor(dy, dt, m.B, m.Cout, m.Tp));
    SC_TRY(check_tensor(x, dt, m.B, m.Cin, m.T));
    SC_TRY(check_tensor(y, dt, m.B, m.Cout, m.Tp));
    SC_TRY(check_tensor(dx, dt, m.B, m.Cin, m.T));
    if (dx_add) SC_TRY(check_tensor(dx_add, dt, m.B, m.Cin, m.T));
    if (desc->residual != SC_RES_NONE) {
        if (x_res) SC_TRY(check_tensor(x_res, dt, m.B, m.Cres, m.Tp));
        else if (m.s != 1 || m.Cres != m.Cin) return SC_ERR_UNSUPPORTED;
        if (dx_res) SC_TRY(check_tensor(dx_res, dt, m.B, m.Cres, m.Tp));
        else if (m.s != 1 || m.Cres != m.Cin) return SC_ERR_UNSUPPORTED;
        // folding the residual path's gradient into dx is only meaningful when the residual source is x itself
        else if (x_res && x_res->ptr != x->ptr) return SC_ERR_UNSUPPORTED;
    }
    SC_TRY(check_params(desc, params));
    SC_TRY(check_saved(desc, saved, false));
    SC_TRY(check_grads(desc, grads));
    if (!workspace) return SC_ERR_WORKSPACE;
    Packed pk;
    if (ctx->gemm_mode == 0) pk = plan_packed(desc, m);
    const Dims& mq = pk.phases ? pk.m : m;
    Bump ws(workspace, workspace_bytes);
    BwdScratch s; BwdPack bp;
    plan_bwd(desc, mq, ws, &s, &ctx->tc);
    if (pk.phases) plan_bwd_pack(desc, pk, ws, &bp);
    if (!ws.ok()) return SC_ERR_WORKSPACE;
    const bool two = pk.phases > 1;
    Prologue pr = length_prologue(m, lengths_dev, s.len_out, s.nvalid, s.blk_off);
    if (two) { pr.phases = pk.phases; pr.len_dense = bp.len_dense; }
    pr.zero = s.gmax; pr.nzero = 1;
    if (needs_w16(desc, m)) pr.convert(params->wp, s.w16, m.Cout * m.Cin);
    prologue(L, pr);
    BwdIO io{};
    io.gmax = s.gmax; io.w16 = s.w16;
    io.dy = dy->ptr; io.x = x->ptr; io.y = y->ptr;
    io.xres = desc->residual != SC_RES_NONE ? (x_res ? x_res->ptr : x->ptr) : nullptr;
    io.dx = dx->ptr; io.dx_res = (desc->residual != SC_RES_NONE && dx_res) ? dx_res->ptr : nullptr;
    io.dx_add = dx_add ? dx_add->ptr : nullptr;
    io.len_in = lengths_dev; io.len_out = s.len_out; io.nvalid = s.nvalid; io.blk_off = s.blk_off;
    io.x_clean = false; io.res_clean = false;
    io.done = ctx->ev[2]; io.fork_early = true;
    sc_block_saved sv = *saved;
    if (pk.phases) {
        // packs what the contractions read; the batch-norm kernels read dy, y, v and vr as they are
        PackList in{}, out{};
        auto add = [&](PackList& l, const void* src, void* dst, int C, const int* len) { l.src[l.count] = src; l.dst[l.count] = dst; l.C[l.count] = C; l.len[l.count] = len; ++l.count; };
        const bool proj = desc->residual == SC_RES_PROJ, own = proj && io.xres == io.x && m.s == 1;
        add(in, io.x, bp.x, m.Cin, lengths_dev);
        if (io.dx_add) { add(in, io.dx_add, bp.dx_add, m.Cin, lengths_dev); io.dx_add = bp.dx_add; }
        const int* len_o = two ? bp.len_dense : s.len_out;
        PackList& o = m.s == 1 ? in : out;               // tensors with output frames share the launch when the frames agree
        if (desc->has_dw) { add(o, sv.u, bp.u, m.Cin, len_o); sv.u = bp.u; }
        if (proj && !own) add(o, io.xres, bp.xres, m.Cres, len_o);
        pack_frames(L, in, m.B, m.T, pk.Tq, pk.phases);
        if (m.s != 1) pack_frames(L, out, m.B, m.Tp, mq.Tp, 1);
        if (proj) io.xres = own ? bp.x : bp.xres;
        io.x = bp.x; io.dx = bp.dx;
        if (io.dx_res) io.dx_res = bp.dx_res;
        io.x_clean = io.res_clean = true;
        if (two) io.len_in = s.len_out;
        io.phases = pk.phases; io.Td = m.Tp; io.total_dense = (uint32_t)m.B * m.Cout * m.Tp;
    }
    SC_TRY(block_bwd_impl(ctx, L, desc, mq, io, params, &sv, grads, accumulate, s));
    if (pk.phases) {
        PackList l{}; l.count = 1; l.src[0] = bp.dx; l.dst[0] = dx->ptr; l.C[0] = m.Cin; l.len[0] = lengths_dev;
        if (io.dx_res && m.s == 1) { l.count = 2; l.src[1] = bp.dx_res; l.dst[1] = dx_res->ptr; l.C[1] = m.Cres; l.len[1] = lengths_dev; }
        unpack_frames(L, l, m.B, m.T, pk.Tq, pk.phases);
        if (io.dx_res && m.s != 1) {
            PackList r{}; r.count = 1; r.src[0] = bp.dx_res; r.dst[0] = dx_res->ptr; r.C[0] = m.Cres; r.len[0] = s.len_out;
            unpack_frames(L, r, m.B, m.Tp, mq.Tp, 1);
        }
    }
    wait_side(ctx, L, ctx->ev[2]);
    return finish(ctx);
}
}  // namespace

int sepconv_bwd(sc_ctx* ctx, const sc_block_desc* desc, const sc_tensor* dy, const sc_tensor* x,
                const sc_tensor* x_res, const sc_tensor* y, const int32_t* lengths_dev,
                const sc_block_params* params, const sc_block_saved* saved, sc_tensor* dx,
                sc_tensor* dx_res, const sc_tensor* dx_add, sc_block_grads* grads, int accumulate,
                void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!ctx || !lengths_dev || !desc) return SC_ERR_NULL;
    CallKey& k = ctx->key;
    key_begin(ctx, CALL_BWD, workspace, workspace_bytes);
    k.add(desc, sizeof(*desc)); key_tensor(k, dy); key_tensor(k, x); key_tensor(k, x_res); key_tensor(k, y); k.val(lengths_dev);
    k.add(params, sizeof(*params)); k.add(saved, sizeof(*saved)); key_tensor(k, dx); key_tensor(k, dx_res); key_tensor(k, dx_add);
    k.add(grads, sizeof(*grads)); k.val(accumulate);
    return run_call(ctx, cuda_stream, [&](const Launch& L) { return bwd_call(ctx, L, desc, dy, x, x_res, y, lengths_dev, params, saved, dx, dx_res, dx_add,
                        grads, accumulate, workspace, workspace_bytes); });
}

// ---- encoder ---------------------------------------------------------------------------------
namespace {
struct LayerPlan {
    sc_block_desc d; Dims m;
    sc_block_saved sv; void* y; int* len_out; int* nvalid; int* blk_off; void* w16;
    bool own_lengths;
};
// Backward layer i works in scratch region i % kScratchRegions: its weight-gradient kernels (side stream) may still
// read their operands while the next layers already write their own, and the main stream waits for them only when it
// comes back to the region, kScratchRegions layers later.  (Three regions measured slower than two: weight gradients
// that may lag two layers behind take SMs from the critical path more often than the wait costs.)
constexpr int kScratchRegions = 2;
struct EncPlan {
    std::vector<LayerPlan> L;
    void* gbuf[2];
    std::vector<void*> pend;       // per layer: where the residual gradients for that layer's input collect (or null)
    void* pend_tmp;                // a second residual gradient for a source that already holds one lands here first
    float* gmax_all;               // one |gv| bound per layer, zeroed by one memset at the start of the call
    size_t bytes;
    size_t scratch_mark;           // offset where the shared per-layer scratch starts
    size_t scratch_size;           // its size; kScratchRegions regions of that size in all (backward layers rotate)
    // An input whose row lengths the tensor-core kernels cannot take runs on rows padded to T_pad frames: the frames past a
    // sample's length are masked anyway, so only the call's own tensors are copied (x and dlogits in, logits and dx out).
    int T_pad = 0, T_out = 0;      // 0: not padded; frames of the last layer's dense output
    void *x_pad, *dlogits_pad, *logits_pad, *dx_pad;
};

// Row length for a padded pass (0: none needed): the stride product times 8, so that every layer's rows are whole vectors.
int encoder_pad(const sc_encoder_desc* e) {
    if (e->layers[0].io_dtype == SC_F32) return 0;
    int t = e->layers[0].T_in, div = 8;
    if (t < 1) return 0;
    bool fits = t % 8 == 0;
    for (int i = 0; i < e->n_layers; ++i) {
        const sc_block_desc& d = e->layers[i];
        const int s = (d.has_dw || d.full_conv) ? d.stride : 1;
        if (s != 1 && s != 2) return 0;
        t = (t - 1) / s + 1;
        fits &= t % 8 == 0;
        if (div > (1 << 16)) return 0;
        div *= s;
    }
    if (fits) return 0;
    const int T = e->layers[0].T_in, Tq = (T + div - 1) / div * div;
    const sc_block_desc &f = e->layers[0], &l = e->layers[e->n_layers - 1];
    return (long long)f.B * std::max(f.C_in, l.C_out) * Tq < (1ll << 31) ? Tq : 0;      // the copies index with 32 bits
}

int plan_encoder(const sc_encoder_desc* e, void* base, size_t cap, EncPlan* P, const TcState* tc, bool pad) {
    if (!e || !e->layers || e->n_layers < 1) return SC_ERR_NULL;
    Bump ws(base, cap);
    P->L.resize(e->n_layers);
    int B = e->layers[0].B, T = e->layers[0].T_in, C = e->layers[0].C_in;
    P->T_pad = pad ? encoder_pad(e) : 0;
    if (P->T_pad) {
        P->T_out = T;
        for (int i = 0; i < e->n_layers; ++i)
            P->T_out = (P->T_out - 1) / ((e->layers[i].has_dw || e->layers[i].full_conv) ? e->layers[i].stride : 1) + 1;
        T = P->T_pad;
    }
    size_t max_act = 0, max_res = 0;
    // Residual spans [source, layer]: the residual path's gradient waits in a pending buffer from the backward step of
    // `layer` down to that of `source`.  Spans that do not overlap share a buffer (the five blocks of the QuartzNet
    // encoder use one); spans that overlap or nest get buffers of their own; several layers may share a source (their
    // gradients are summed in the source's buffer).
    const int nl = e->n_layers;
    std::vector<int> last_user(nl, -1), users(nl, 0);
    std::vector<size_t> res_bytes(nl, 0);
    for (int i = 0; i < nl; ++i) {
        if (e->layers[i].residual == SC_RES_NONE || !e->res_from || e->res_from[i] < 0 || e->res_from[i] == i) continue;
        if (e->res_from[i] > i) return SC_ERR_UNSUPPORTED;
        last_user[e->res_from[i]] = i; ++users[e->res_from[i]];
    }
    for (int i = 0; i < e->n_layers; ++i) {
        LayerPlan& lp = P->L[i];
        lp.d = e->layers[i];
        lp.d.B = B; lp.d.T_in = T;
        if (lp.d.C_in != C) return SC_ERR_DIM_INCOMPATIBLE;
        if (lp.d.io_dtype != e->layers[0].io_dtype) return SC_ERR_INCOMPATIBLE;
        if (lp.d.residual != SC_RES_NONE) {
            int j = e->res_from ? e->res_from[i] : -1;
            if (j < 0) j = i;
            if (j > i) return SC_ERR_UNSUPPORTED;
            lp.d.C_res = e->layers[j].C_in;
        }
        SC_TRY(desc_dims(&lp.d, &lp.m));
        const Dims& m = lp.m;
        const size_t es = esize(lp.d.io_dtype);
        if (lp.d.residual != SC_RES_NONE) {
            int j = (e->res_from && e->res_from[i] >= 0) ? e->res_from[i] : i;
            if (P->L[j].m.T != m.Tp) return SC_ERR_UNSUPPORTED;
            max_res = std::max(max_res, es * m.B * m.Cres * m.Tp);
            if (j != i) res_bytes[j] = es * m.B * m.Cres * m.Tp;
        }
        lp.own_lengths = (i == 0) || (m.s != 1);
        if (lp.own_lengths) {
            lp.len_out = (int*)ws.take(sizeof(int) * B); lp.nvalid = (int*)ws.take(sizeof(int));
            lp.blk_off = (int*)ws.take(sizeof(int) * (B + 1));
        } else { lp.len_out = P->L[i - 1].len_out; lp.nvalid = P->L[i - 1].nvalid; lp.blk_off = P->L[i - 1].blk_off; }
        memset(&lp.sv, 0, sizeof(lp.sv));
        if (lp.d.has_dw) lp.sv.u = ws.take(es * B * m.Cin * m.Tp);
        else if (i == 0) lp.sv.u = ws.take(es * B * m.Cin * m.Tp);
        if (lp.d.has_bn) {
            lp.sv.v = ws.take(dtype_size(ntype_of(lp.d.io_dtype)) * B * m.Cout * m.Tp);
            lp.sv.mean = (float*)ws.take(4 * m.Cout); lp.sv.invstd = (float*)ws.take(4 * m.Cout);
        }
        if (lp.d.residual == SC_RES_PROJ) {
            lp.sv.vr = ws.take(dtype_size(ntype_of(lp.d.io_dtype)) * B * m.Cout * m.Tp);
            lp.sv.mean_r = (float*)ws.take(4 * m.Cout); lp.sv.invstd_r = (float*)ws.take(4 * m.Cout);
        }
        lp.y = (i + 1 < e->n_layers) ? ws.take(es * B * m.Cout * m.Tp) : nullptr;
        lp.w16 = (op_dtype(&lp.d) != lp.d.io_dtype) ? ws.take((size_t)2 * m.Cout * m.Cin) : nullptr;
        max_act = std::max(max_act, es * B * (size_t)m.Cin * m.T);
        max_act = std::max(max_act, es * B * (size_t)m.Cout * m.Tp);
        C = m.Cout; T = m.Tp;
    }
    // shared scratch: plan every layer from the same offset and keep the maximum
    const size_t mark = ws.off;
    size_t hi = mark;
    for (int i = 0; i < e->n_layers; ++i) {
        Bump b(base, cap); b.off = mark; FwdScratch f; plan_fwd(&P->L[i].d, P->L[i].m, b, &f, tc); hi = std::max(hi, b.off);
        Bump c(base, cap); c.off = mark; BwdScratch s; plan_bwd(&P->L[i].d, P->L[i].m, c, &s, tc); hi = std::max(hi, c.off);
    }
    hi = (hi + 255) & ~(size_t)255;
    ws.off = hi + (size_t)(kScratchRegions - 1) * (hi - mark);
    P->scratch_size = hi - mark;
    P->gbuf[0] = ws.take(max_act); P->gbuf[1] = ws.take(max_act);
    {
        // interval colouring in source order: a buffer whose span ended strictly before this source is free again
        struct Buf { int end; size_t bytes; };
        std::vector<Buf> bufs;
        std::vector<int> colour(nl, -1);
        bool need_tmp = false;
        for (int j = 0; j < nl; ++j) {
            if (last_user[j] < 0) continue;
            if (users[j] > 1) need_tmp = true;
            int c = -1;
            for (size_t q = 0; q < bufs.size(); ++q) if (bufs[q].end < j) { c = (int)q; break; }
            if (c < 0) { bufs.push_back(Buf{0, 0}); c = (int)bufs.size() - 1; }
            bufs[c].end = last_user[j]; bufs[c].bytes = std::max(bufs[c].bytes, res_bytes[j]);
            colour[j] = c;
        }
        std::vector<void*> addr(bufs.size(), nullptr);
        for (size_t q = 0; q < bufs.size(); ++q) addr[q] = ws.take(bufs[q].bytes);
        P->pend.assign(nl, nullptr);
        for (int j = 0; j < nl; ++j) if (colour[j] >= 0) P->pend[j] = addr[colour[j]];
        P->pend_tmp = need_tmp ? ws.take(max_res) : nullptr;
    }
    P->gmax_all = (float*)ws.take(sizeof(float) * e->n_layers);
    if (P->T_pad) {
        const LayerPlan &f = P->L[0], &l = P->L[nl - 1];
        const size_t es = esize(f.d.io_dtype), in = es * f.m.B * f.m.Cin * f.m.T, out = es * l.m.B * l.m.Cout * l.m.Tp;
        P->x_pad = ws.take(in); P->dx_pad = ws.take(in); P->logits_pad = ws.take(out); P->dlogits_pad = ws.take(out);
    }
    P->bytes = ws.off + 256;
    if (!ws.ok()) return SC_ERR_WORKSPACE;
    P->scratch_mark = mark;
    return SC_OK;
}

sc_block_params layer_params(const void* blob, const int64_t* off) {
    auto at = [&](int j) -> const void* { return off[j] < 0 ? nullptr : (const char*)blob + off[j]; };
    sc_block_params p;
    p.wd = at(0); p.wp = at(1); p.gamma = (const float*)at(2); p.beta = (const float*)at(3);
    p.bias = (const float*)at(4); p.wr = at(5); p.gamma_r = (const float*)at(6); p.beta_r = (const float*)at(7);
    return p;
}
sc_block_grads layer_grads(void* blob, const int64_t* off) {
    auto at = [&](int j) -> float* { return off[j] < 0 ? nullptr : (float*)((char*)blob + off[j]); };
    sc_block_grads g;
    g.dwd = at(0); g.dwp = at(1); g.dgamma = at(2); g.dbeta = at(3); g.dbias = at(4);
    g.dwr = at(5); g.dgamma_r = at(6); g.dbeta_r = at(7);
    return g;
}
// one tensor in (pack) or out (unpack) of padded rows
void copy_frames(const Launch& L, bool in, const void* src, void* dst, int C, const int* len, int B, int T, int Tq) {
    PackList l{}; l.count = 1; l.src[0] = src; l.dst[0] = dst; l.C[0] = C; l.len[0] = len;
    if (in) pack_frames(L, l, B, T, Tq, 1); else unpack_frames(L, l, B, T, Tq, 1);
}
// whether a layer after the first changes the lengths again
bool strided_later(const EncPlan& P) {
    for (size_t i = 1; i < P.L.size(); ++i) if (P.L[i].own_lengths) return true;
    return false;
}
// Lengths of the first layer (the encoder's, unless a later layer strides too), float16 copies of the pointwise weights of
// every layer that needs one and, for a training pass, the zeroed |gv| bounds.
void encoder_prologue(const Launch& L, const sc_encoder_desc* e, const EncPlan& P, const int* lengths, int* out_lengths,
                      const void* blob, const int64_t* offs, bool train) {
    const LayerPlan& f = P.L[0];
    Prologue pr = length_prologue(f.m, lengths, f.len_out, f.nvalid, f.blk_off);
    pr.T_in = e->layers[0].T_in;                  // the legal range, whatever the rows are padded to
    if (!strided_later(P)) pr.len_user = out_lengths;
    if (train) { pr.zero = P.gmax_all; pr.nzero = e->n_layers; }
    for (int i = 0; i < e->n_layers; ++i) {
        const LayerPlan& l = P.L[i];
        if (!l.w16) continue;
        if (pr.conv.count == kMaxConvert) { Prologue more; std::swap(more.conv, pr.conv); prologue(L, more); }
        pr.convert(layer_params(blob, offs + 8 * i).wp, l.w16, l.m.Cout * l.m.Cin);
    }
    prologue(L, pr);
}
}  // namespace

int encoder_workspace_bytes(const sc_encoder_desc* desc, size_t* bytes) {
    if (!bytes) return SC_ERR_NULL;
    EncPlan P;
    SC_TRY(plan_encoder(desc, nullptr, 0, &P, nullptr, true));
    *bytes = P.bytes;
    if (P.T_pad) { SC_TRY(plan_encoder(desc, nullptr, 0, &P, nullptr, false)); *bytes = std::max(*bytes, P.bytes); }
    return SC_OK;
}

int encoder_infer_workspace_bytes(const sc_encoder_desc* desc, size_t* bytes) {
    return encoder_workspace_bytes(desc, bytes);      // the same plan: per-layer buffers double as scratch
}

namespace {
int encoder_infer_call(sc_ctx* ctx, const Launch& L, const sc_encoder_desc* e, const sc_tensor* x, const int32_t* lengths_dev,
                       const void* params_blob, const int64_t* param_offsets, const void* running_blob,
                       const int64_t* running_offsets, sc_tensor* out, int32_t* out_lengths_dev, void* workspace,
                       size_t workspace_bytes) {
    if (!workspace) return SC_ERR_WORKSPACE;
    EncPlan P;
    SC_TRY(plan_encoder(e, workspace, workspace_bytes, &P, &ctx->tc, ctx->gemm_mode == 0));
    const int n = e->n_layers;
    const Dims& m0 = P.L[0].m; const Dims& ml = P.L[n - 1].m;
    const int dt = P.L[0].d.io_dtype;
    const int T_in = e->layers[0].T_in;
    SC_TRY(check_tensor(x, dt, m0.B, m0.Cin, T_in));
    SC_TRY(check_tensor(out, dt, ml.B, ml.Cout, P.T_pad ? P.T_out : ml.Tp));
    auto stat = [&](int i, int j) -> const float* {
        const int64_t o = running_offsets[4 * i + j];
        return o < 0 ? nullptr : (const float*)((const char*)running_blob + o);
    };
    for (int i = 0; i < n; ++i) {
        const sc_block_params prm = layer_params(params_blob, param_offsets + 8 * i);
        SC_TRY(check_params(&P.L[i].d, &prm));
        if (P.L[i].d.has_bn && (!stat(i, 0) || !stat(i, 1))) return SC_ERR_NULL;
        if (P.L[i].d.residual == SC_RES_PROJ && (!stat(i, 2) || !stat(i, 3))) return SC_ERR_NULL;
    }
    encoder_prologue(L, e, P, lengths_dev, out_lengths_dev, params_blob, param_offsets, false);
    const void* x_in = x->ptr;
    void* y_out = out->ptr;
    if (P.T_pad) { copy_frames(L, true, x->ptr, P.x_pad, m0.Cin, lengths_dev, m0.B, T_in, m0.T); x_in = P.x_pad; y_out = P.logits_pad; }
    auto input_of = [&](int i) -> const void* { return i == 0 ? x_in : P.L[i - 1].y; };
    auto res_src = [&](int i) -> int { return (e->res_from && e->res_from[i] >= 0) ? e->res_from[i] : i; };
    for (int i = 0; i < n; ++i) {
        LayerPlan& lp = P.L[i];
        sc_block_params prm = layer_params(params_blob, param_offsets + 8 * i);
        InferStats inf{stat(i, 0), stat(i, 1), stat(i, 2), stat(i, 3)};
        Bump b(workspace, workspace_bytes); b.off = P.scratch_mark;
        FwdScratch f; plan_fwd(&lp.d, lp.m, b, &f, &ctx->tc);
        BlockIO io{};
        io.x = input_of(i);
        io.xres = lp.d.residual != SC_RES_NONE ? input_of(res_src(i)) : nullptr;
        io.y = (i + 1 < n) ? lp.y : y_out;
        io.len_in = i == 0 ? lengths_dev : P.L[i - 1].len_out; io.len_out = lp.len_out; io.nvalid = lp.nvalid; io.blk_off = lp.blk_off;
        io.x_clean = i > 0; io.res_clean = lp.d.residual != SC_RES_NONE && res_src(i) > 0;
        io.lengths_ready = i == 0 || !lp.own_lengths;
        io.w16 = lp.w16;
        if (P.T_pad) io.x_clean = true;
        SC_TRY(block_fwd_impl(ctx, L, &lp.d, lp.m, io, &prm, &lp.sv, nullptr, nullptr, f, &inf));
    }
    if (P.T_pad) copy_frames(L, false, P.logits_pad, out->ptr, ml.Cout, P.L[n - 1].len_out, ml.B, P.T_out, ml.Tp);
    if (out_lengths_dev && strided_later(P))
        cudaMemcpyAsync(out_lengths_dev, P.L[n - 1].len_out, sizeof(int) * m0.B, cudaMemcpyDeviceToDevice, L.stream);
    return finish(ctx);
}
}  // namespace

int encoder_infer(sc_ctx* ctx, const sc_encoder_desc* e, const sc_tensor* x, const int32_t* lengths_dev,
                  const void* params_blob, const int64_t* param_offsets, const void* running_blob,
                  const int64_t* running_offsets, sc_tensor* out, int32_t* out_lengths_dev, void* workspace,
                  size_t workspace_bytes, void* cuda_stream) {
    if (!ctx || !lengths_dev || !params_blob || !param_offsets || !running_blob || !running_offsets) return SC_ERR_NULL;
    if (!e || !e->layers || e->n_layers < 1) return SC_ERR_NULL;
    CallKey& k = ctx->key;
    key_begin(ctx, CALL_ENC_INFER, workspace, workspace_bytes);
    k.val(e->n_layers); k.add(e->layers, sizeof(sc_block_desc) * e->n_layers); k.add(e->res_from, e->res_from ? sizeof(int32_t) * e->n_layers : 0);
    key_tensor(k, x); k.val(lengths_dev); k.val(params_blob); k.add(param_offsets, sizeof(int64_t) * 8 * e->n_layers);
    k.val(running_blob); k.add(running_offsets, sizeof(int64_t) * 4 * e->n_layers); key_tensor(k, out); k.val(out_lengths_dev);
    return run_call(ctx, cuda_stream, [&](const Launch& L) { return encoder_infer_call(ctx, L, e, x, lengths_dev, params_blob, param_offsets, running_blob,
                                  running_offsets, out, out_lengths_dev, workspace, workspace_bytes); });
}

namespace {
int encoder_call(sc_ctx* ctx, const Launch& L, const sc_encoder_desc* e, const sc_tensor* x, const int32_t* lengths_dev,
                         const void* params_blob, const int64_t* param_offsets, const sc_tensor* dlogits,
                         sc_tensor* logits, int32_t* out_lengths_dev, void* grads_blob,
                         const int64_t* grad_offsets, sc_tensor* dx, int accumulate, void* workspace,
                         size_t workspace_bytes) {
    if (!workspace) return SC_ERR_WORKSPACE;
    EncPlan P;
    SC_TRY(plan_encoder(e, workspace, workspace_bytes, &P, &ctx->tc, ctx->gemm_mode == 0));
    const int n = e->n_layers;
    const size_t mark = P.scratch_mark;
    const Dims& m0 = P.L[0].m; const Dims& ml = P.L[n - 1].m;
    const int dt = P.L[0].d.io_dtype;
    const int T_in = e->layers[0].T_in, T_out = P.T_pad ? P.T_out : ml.Tp;
    SC_TRY(check_tensor(x, dt, m0.B, m0.Cin, T_in));
    SC_TRY(check_tensor(logits, dt, ml.B, ml.Cout, T_out));
    SC_TRY(check_tensor(dlogits, dt, ml.B, ml.Cout, T_out));
    if (dx) SC_TRY(check_tensor(dx, dt, m0.B, m0.Cin, T_in));
    std::vector<sc_block_params> prm(n);
    std::vector<sc_block_grads> grd(n);
    for (int i = 0; i < n; ++i) {
        prm[i] = layer_params(params_blob, param_offsets + 8 * i);
        grd[i] = layer_grads(grads_blob, grad_offsets + 8 * i);
        SC_TRY(check_params(&P.L[i].d, &prm[i]));
        SC_TRY(check_grads(&P.L[i].d, &grd[i]));
    }
    const void *x_in = x->ptr, *dl = dlogits->ptr;
    void *lg = logits->ptr, *dx_out = dx ? dx->ptr : nullptr;
    // ahead of the copies: the first layer's contraction reads the block offsets before it waits, so a kernel has to lie between
    encoder_prologue(L, e, P, lengths_dev, out_lengths_dev, params_blob, param_offsets, true);
    if (P.T_pad) {
        copy_frames(L, true, x->ptr, P.x_pad, m0.Cin, lengths_dev, m0.B, T_in, m0.T);
        copy_frames(L, true, dlogits->ptr, P.dlogits_pad, ml.Cout, nullptr, ml.B, T_out, ml.Tp);
        x_in = P.x_pad; dl = P.dlogits_pad; lg = P.logits_pad; if (dx) dx_out = P.dx_pad;
    }
    auto input_of = [&](int i) -> const void* { return i == 0 ? x_in : P.L[i - 1].y; };
    auto len_in_of = [&](int i) -> const int* { return i == 0 ? lengths_dev : P.L[i - 1].len_out; };
    auto res_src = [&](int i) -> int { return (e->res_from && e->res_from[i] >= 0) ? e->res_from[i] : i; };

    // forward
    for (int i = 0; i < n; ++i) {
        LayerPlan& lp = P.L[i];
        Bump b(workspace, workspace_bytes); b.off = mark;
        FwdScratch f; plan_fwd(&lp.d, lp.m, b, &f, &ctx->tc);
        BlockIO io{};
        io.x = input_of(i);
        io.xres = lp.d.residual != SC_RES_NONE ? input_of(res_src(i)) : nullptr;
        io.y = (i + 1 < n) ? lp.y : lg;
        io.len_in = len_in_of(i); io.len_out = lp.len_out; io.nvalid = lp.nvalid; io.blk_off = lp.blk_off;
        io.x_clean = i > 0 || P.T_pad; io.res_clean = lp.d.residual != SC_RES_NONE && res_src(i) > 0;
        io.lengths_ready = i == 0 || !lp.own_lengths;
        io.w16 = lp.w16;
        SC_TRY(block_fwd_impl(ctx, L, &lp.d, lp.m, io, &prm[i], &lp.sv, nullptr, nullptr, f));
    }
    if (out_lengths_dev && strided_later(P))
        cudaMemcpyAsync(out_lengths_dev, P.L[n - 1].len_out, sizeof(int) * m0.B, cudaMemcpyDeviceToDevice, L.stream);

    if (P.T_pad) copy_frames(L, false, lg, logits->ptr, ml.Cout, P.L[n - 1].len_out, ml.B, T_out, ml.Tp);

    // backward
    const void* g = dl;
    std::vector<char> has_pending(n, 0);
    bool side_busy[kScratchRegions] = {};
    cudaEvent_t done_ev[3] = {ctx->ev[2], ctx->ev[3], ctx->ev[6]};
    for (int i = n - 1; i >= 0; --i) {
        LayerPlan& lp = P.L[i];
        // this layer reuses the scratch region of layer i + kScratchRegions: that layer's side-stream kernels must be done
        const int region = i % kScratchRegions;
        if (side_busy[region]) wait_side(ctx, L, done_ev[region]);
        Bump b(workspace, workspace_bytes); b.off = mark + (size_t)region * P.scratch_size;
        BwdScratch s; plan_bwd(&lp.d, lp.m, b, &s, &ctx->tc);
        BwdIO io{};
        io.done = done_ev[region]; side_busy[region] = true;
        io.dy = g; io.x = input_of(i); io.y = (i + 1 < n) ? lp.y : lg;
        io.xres = lp.d.residual != SC_RES_NONE ? input_of(res_src(i)) : nullptr;
        io.dx = (i == 0) ? dx_out : P.gbuf[i & 1];
        io.dx_res = nullptr;
        const int src = res_src(i);
        const bool to_pending = lp.d.residual != SC_RES_NONE && src != i;
        const bool second = to_pending && has_pending[src];       // the source's buffer already holds a gradient
        if (to_pending) { io.dx_res = second ? P.pend_tmp : P.pend[src]; has_pending[src] = 1; }
        io.dx_add = has_pending[i] ? P.pend[i] : nullptr;
        io.len_in = len_in_of(i); io.len_out = lp.len_out; io.nvalid = lp.nvalid; io.blk_off = lp.blk_off;
        io.x_clean = i > 0 || P.T_pad; io.res_clean = lp.d.residual != SC_RES_NONE && res_src(i) > 0;
        io.w16 = lp.w16;
        io.gmax = P.gmax_all + i;
        SC_TRY(block_bwd_impl(ctx, L, &lp.d, lp.m, io, &prm[i], &lp.sv, &grd[i], accumulate, s));
        if (second)
            ew_add_masked(L, dt, P.pend[src], P.pend[src], P.pend_tmp, nullptr, len_in_of(src), P.L[src].m.B, P.L[src].m.Cin, P.L[src].m.T);
        g = io.dx;
    }
    if (P.T_pad && dx) copy_frames(L, false, dx_out, dx->ptr, m0.Cin, lengths_dev, m0.B, T_in, m0.T);
    for (int q = 0; q < kScratchRegions; ++q) if (side_busy[q]) wait_side(ctx, L, done_ev[q]);     // join before returning
    return finish(ctx);
}
}  // namespace

int encoder_fwd_bwd(sc_ctx* ctx, const sc_encoder_desc* e, const sc_tensor* x, const int32_t* lengths_dev,
                    const void* params_blob, const int64_t* param_offsets, const sc_tensor* dlogits,
                    sc_tensor* logits, int32_t* out_lengths_dev, void* grads_blob,
                    const int64_t* grad_offsets, sc_tensor* dx, int accumulate, void* workspace,
                    size_t workspace_bytes, void* cuda_stream) {
    if (!ctx || !lengths_dev || !params_blob || !param_offsets || !grads_blob || !grad_offsets) return SC_ERR_NULL;
    if (!e || !e->layers || e->n_layers < 1) return SC_ERR_NULL;
    CallKey& k = ctx->key;
    key_begin(ctx, CALL_ENC, workspace, workspace_bytes);
    k.val(e->n_layers); k.add(e->layers, sizeof(sc_block_desc) * e->n_layers); k.add(e->res_from, e->res_from ? sizeof(int32_t) * e->n_layers : 0);
    key_tensor(k, x); k.val(lengths_dev); k.val(params_blob); k.add(param_offsets, sizeof(int64_t) * 8 * e->n_layers);
    key_tensor(k, dlogits); key_tensor(k, logits); k.val(out_lengths_dev); k.val(grads_blob);
    k.add(grad_offsets, sizeof(int64_t) * 8 * e->n_layers); key_tensor(k, dx); k.val(accumulate);
    return run_call(ctx, cuda_stream, [&](const Launch& L) { return encoder_call(ctx, L, e, x, lengths_dev, params_blob, param_offsets, dlogits, logits,
                                    out_lengths_dev, grads_blob, grad_offsets, dx, accumulate, workspace, workspace_bytes); });
}

}  // extern "C"

int sc::fwd_direct(sc_ctx* ctx, const sc_block_desc* desc, const sc_tensor* x, const sc_tensor* x_res, const int32_t* lengths_dev,
                   const sc_block_params* params, sc_tensor* y, int32_t* out_lengths_dev, sc_block_saved* saved, void* workspace,
                   size_t workspace_bytes, void* cuda_stream) {
    if (!ctx || !lengths_dev) return SC_ERR_NULL;
    return fwd_call(ctx, Launch{(cudaStream_t)cuda_stream, ctx->status_dev, &ctx->launches, &ctx->prof, ctx->gemm_mode, ctx->pdl, ctx->fresh}, desc, x,
                    x_res, lengths_dev, params, y, out_lengths_dev, saved, nullptr, nullptr, workspace, workspace_bytes, true);
}

int sc::fwd_dense_bytes(const sc_block_desc* desc, size_t* bytes) {
    Dims m;
    SC_TRY(desc_dims(desc, &m));
    Bump b(nullptr, 0); FwdScratch f; plan_fwd(desc, m, b, &f, nullptr, false);
    *bytes = b.off + 256;
    return SC_OK;
}
