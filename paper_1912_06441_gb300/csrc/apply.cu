// Operator application (Eq. general_do) and the RK4 driver (Sec. 5.1).
//
// Both are streaming gather-sums over the stencils: per stencil entry e of node i, read
// col[e] and the weights w[e][*] once (HBM), gather f[col[e]] (stays in L2: the field is
// small next to the weight stream and nodes are numbered in spatial order), and accumulate
// (f_j - f_i) w.
//
// The apply and the stages on float fields read the CSR rows: a group of G lanes shares one node, the
// lanes read consecutive entries, so every weight and index load of a warp is a contiguous, fully used
// segment; UNR entries per lane are in flight before the first use.  The partial sums of a group are combined with
// shuffles: by a reduce-scatter over the operators in the apply (each lane ends with one
// operator's sum), by a butterfly tree in the stages.  (G, UNR) is chosen per context by a small autotuner: the first
// apply (or run) for a given operator count, data types and problem class times every shape once on the real
// stencils and keeps the fastest.
//
// The stages on double fields read combined weights in the sliced layout of sell.cu: the FP64 pipe bounds them, and
// there the lanes that combine sums and update nodes are a few percent of its work.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "df64.cuh"
#include "sell_fill.cuh"

namespace labfm {
namespace {

constexpr int APPLY_THREADS = 256;

// Weights of entry e (NOPS of them) into wv[], converted to the accumulation type.
template <int NOPS, class WT, class AT>
__device__ __forceinline__ void load_w(const WT *__restrict__ w, int64_t e, AT *wv)
{
    const WT *p = w + e * NOPS;
    if constexpr (NOPS == 4 && sizeof(WT) == 8) {
        double2 a = __ldcs(reinterpret_cast<const double2 *>(p));
        double2 b = __ldcs(reinterpret_cast<const double2 *>(p) + 1);
        wv[0] = (AT)a.x; wv[1] = (AT)a.y; wv[2] = (AT)b.x; wv[3] = (AT)b.y;
    } else if constexpr (NOPS == 4 && sizeof(WT) == 4) {
        float4 a = __ldcs(reinterpret_cast<const float4 *>(p));
        wv[0] = (AT)a.x; wv[1] = (AT)a.y; wv[2] = (AT)a.z; wv[3] = (AT)a.w;
    } else if constexpr (NOPS == 2 && sizeof(WT) == 8) {
        double2 a = __ldcs(reinterpret_cast<const double2 *>(p));
        wv[0] = (AT)a.x; wv[1] = (AT)a.y;
    } else {
#pragma unroll
        for (int d = 0; d < NOPS; d++) wv[d] = (AT)__ldcs(p + d);
    }
}

template <class FT, class WT>
using acc_t = typename std::conditional<std::is_same<FT, float>::value && std::is_same<WT, float>::value, float,
                                        double>::type;

// out[sel(d)][i] = sum_j (f_j - f_i) w_ji^d for the operators in mask.
template <int NOPS, class FT, class WT, int UNR>
__global__ void __launch_bounds__(APPLY_THREADS) k_apply(int64_t n, const int64_t *__restrict__ row_ptr,
                                                         const int32_t *__restrict__ col, const WT *__restrict__ w,
                                                         const FT *__restrict__ f, FT *__restrict__ out, uint32_t mask,
                                                         int lg_g)
{
    using AT = acc_t<FT, WT>;
    const int G = 1 << lg_g;  // lanes per node, a power of two
    const int lane = threadIdx.x & (G - 1);
    const int64_t i = ((int64_t)blockIdx.x * APPLY_THREADS + threadIdx.x) >> lg_g;
    const bool live = i < n;
    int64_t rs = 0, re = 0;
    AT fi = 0;
    if (live) {
        rs = row_ptr[i];
        re = row_ptr[i + 1];
        fi = (AT)__ldg(f + i);
    }
    AT acc[NOPS];
#pragma unroll
    for (int d = 0; d < NOPS; d++) acc[d] = 0;
    for (int64_t base = rs; base < re; base += (int64_t)G * UNR) {
        int cj[UNR];
        AT wv[UNR][NOPS];
#pragma unroll
        for (int u = 0; u < UNR; u++) {
            int64_t e = base + (int64_t)u * G + lane;
            if (e < re) {
                cj[u] = __ldcs(col + e);
                load_w<NOPS>(w, e, wv[u]);
            } else {
                cj[u] = -1;
#pragma unroll
                for (int d = 0; d < NOPS; d++) wv[u][d] = 0;
            }
        }
#pragma unroll
        for (int u = 0; u < UNR; u++) {
            if (cj[u] >= 0) {
                AT df = (AT)__ldg(f + cj[u]) - fi;
#pragma unroll
                for (int d = 0; d < NOPS; d++) acc[d] = fma(df, wv[u][d], acc[d]);
            }
        }
    }
    // Reduce-scatter over the node's G lanes (G >= NP, NOPS padded to the power of two NP): at
    // offsets G/2, G/4, ... each lane keeps one half of its operators and adds the partner's
    // half, until it holds one operator's partial, d = lane / (G / NP); the remaining offsets
    // add that one value.  NP - 1 + log2(G / NP) adds per lane instead of NOPS log2(G) (FP64
    // adds are scarce), in a fixed order.
    constexpr int NP = NOPS <= 1 ? 1 : NOPS <= 2 ? 2 : NOPS <= 4 ? 4 : 8;
    AT v[NP];
#pragma unroll
    for (int d = 0; d < NP; d++) v[d] = d < NOPS ? acc[d] : (AT)0;
    int o = G >> 1;
#pragma unroll
    for (int m = NP; m > 1; m >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < m / 2; j++) {
            const AT send = upper ? v[j] : v[j + m / 2];
            const AT keep = upper ? v[j + m / 2] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    const int per = G / NP;  // lanes holding the same operator's sum
    const int d = lane / per;
    if (live && (lane & (per - 1)) == 0 && d < NOPS && ((mask >> d) & 1u)) {
        const int row = __popc(mask & ((1u << d) - 1u));
        out[(int64_t)row * n + i] = (FT)v[0];
    }
}

// Storage of the combined RK4 weight wc_ji = sum_d beta_d w_ji^d (a context-owned buffer):
//   CW_S64  double                    FP64 weights, FP64 fields: accumulated in double, sliced layout
//   CW_S32  float                     FP32 weights, FP64 fields: accumulated in double, sliced layout
//   CW_F32  int2 (j, w)               FP32 weights and fields: each entry's stencil index and weight as one
//                                     8-byte word in CSR order, accumulated in float
//   CW_DF   int2 (j, hi), float lo    FP64 weights, FP32 fields: the double rounded to a
//                                     double-float pair once, here, so that the stage
//                                     accumulates on the FP32 pipes (about 48 bits, far below the
//                                     FP32 field rounding) instead of converting and multiplying
//                                     in FP64 for every stencil entry; the low parts follow the
//                                     nnz index/high-part words
// Packing the index with the weight gives one wide load per entry for the same bytes.
enum { CW_S64 = 0, CW_F32 = 1, CW_DF = 2, CW_S32 = 3 };

int cw_format(int fdt, int wdt)
{
    if (fdt == LABFM_F64) return wdt == LABFM_F64 ? CW_S64 : CW_S32;
    return wdt == LABFM_F32 ? CW_F32 : CW_DF;
}
bool cw_sliced(int fmt) { return fmt == CW_S64 || fmt == CW_S32; }
size_t cw_bytes(const labfm_ctx *ctx, int fmt)
{
    if (cw_sliced(fmt)) return (fmt == CW_S64 ? 8 : 4) * (size_t)ctx->sell.places;
    return (fmt == CW_DF ? 12 : 8) * (size_t)ctx->nnz;
}

struct Beta {
    double v[MAX_OPS];
};

template <class WT>
__global__ void k_combine(int64_t nnz, int n_ops, const WT *__restrict__ w, const int32_t *__restrict__ col,
                          void *__restrict__ wc, int fmt, Beta b)
{
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nnz) return;
    double s = 0.0;
    for (int d = 0; d < n_ops; d++) s = fma(b.v[d], (double)w[e * n_ops + d], s);
    if (fmt == CW_F32) {
        ((int2 *)wc)[e] = make_int2(col[e], __float_as_int((float)s));
    } else {
        df v = df_from_double(s);
        ((int2 *)wc)[e] = make_int2(col[e], __float_as_int(v.hi));
        ((float *)((int2 *)wc + nnz))[e] = v.lo;
    }
}

// wc of an entry, for the sliced layout
template <class WT>
struct Combined {
    const WT *__restrict__ w;
    int n_ops;
    Beta b;
    __device__ __forceinline__ void operator()(int64_t e, WT *v) const
    {
        double s = 0.0;
        for (int d = 0; d < n_ops; d++) s = fma(b.v[d], (double)w[e * n_ops + d], s);
        v[0] = (WT)s;
    }
};

// One RK4 stage.  F_i = sum_j (src_j - src_i) wc_ji (0 on frozen nodes), then
//   stage 0: acc = u + dt/6 F,  nxt = u + dt/2 F
//   stage 1: acc += dt/3 F,     nxt = u + dt/2 F
//   stage 2: acc += dt/3 F,     nxt = u + dt F
//   stage 3: u = acc + dt/6 F
// On double fields the coefficients are products formed on the host (in FP64 a product per thread takes the pipe as long
// as a stencil entry of the warp).
template <int CW, int UNR>
__global__ void __launch_bounds__(APPLY_THREADS) k_rk4_stage_csr(int64_t n, const int64_t *__restrict__ row_ptr,
                                                             const int32_t *__restrict__ col,
                                                             const void *__restrict__ wc_raw,
                                                             const float *__restrict__ wc_lo,
                                                             const float *__restrict__ src, float *__restrict__ u,
                                                             float *__restrict__ acc_buf, float *__restrict__ nxt,
                                                             const uint8_t *__restrict__ frozen, int stage, float dt,
                                                             int lg_g)
{
    const int2 *__restrict__ wcp = (const int2 *)wc_raw;
    const int G = 1 << lg_g;  // lanes per node, a power of two
    const int lane = threadIdx.x & (G - 1);
    const int64_t i = ((int64_t)blockIdx.x * APPLY_THREADS + threadIdx.x) >> lg_g;
    const bool live = i < n;
    int64_t rs = 0, re = 0;
    float si = 0.0f;
    if (live) {
        rs = row_ptr[i];
        re = row_ptr[i + 1];
        si = src[i];
    }
    float acc = 0.0f;
    df accd{0.0f, 0.0f};
    // FP32 weights: the stencil stream is software-pipelined (the next batch of UNR entries per
    // lane is loaded before the gathers of the current one, so its latency overlaps them: +8 % at
    // 2048^2); with double-float weights the second batch's registers cost more than the overlap
    // gains (-11 %), so those load each batch just before its gathers
    constexpr bool PIPE = CW == CW_F32;
    int cn[UNR];
    float2 wn[UNR];  // (weight, low part)
    auto load_batch = [&](int64_t base) {
#pragma unroll
        for (int q = 0; q < UNR; q++) {
            const int64_t e = base + (int64_t)q * G + lane;
            if (e < re) {
                const int2 pr = __ldcs(wcp + e);  // stencil index and (high part of the) weight
                cn[q] = pr.x;
                wn[q] = make_float2(__int_as_float(pr.y), CW == CW_DF ? __ldcs(wc_lo + e) : 0.0f);
            } else {
                cn[q] = -1;
            }
        }
    };
    if (PIPE && rs < re) load_batch(rs);
    for (int64_t base = rs; base < re; base += (int64_t)G * UNR) {
        if (!PIPE) load_batch(base);
        int cj[UNR];
        float2 wv[UNR];
#pragma unroll
        for (int q = 0; q < UNR; q++) {
            cj[q] = cn[q];
            wv[q] = wn[q];
        }
        if (PIPE && base + (int64_t)G * UNR < re) load_batch(base + (int64_t)G * UNR);
#pragma unroll
        for (int q = 0; q < UNR; q++) {
            if (cj[q] >= 0) {
                if constexpr (CW == CW_DF) {
                    float dh, dl;  // src_j - src_i exactly, as a double-float
                    two_sum(src[cj[q]], -si, dh, dl);
                    accd = df_fma(df{dh, dl}, df{wv[q].x, wv[q].y}, accd);
                } else {
                    acc = fma(src[cj[q]] - si, wv[q].x, acc);
                }
            }
        }
    }
    if constexpr (CW == CW_DF) {
        for (int o = G >> 1; o > 0; o >>= 1) {
            df other{__shfl_xor_sync(0xffffffffu, accd.hi, o), __shfl_xor_sync(0xffffffffu, accd.lo, o)};
            accd = df_add(accd, other);
        }
        acc = accd.hi + accd.lo;
    } else {
        for (int o = G >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if (!live || lane != 0) return;
    const float F = (frozen && frozen[i]) ? 0.0f : acc;
    const float ui = u[i];
    switch (stage) {
    case 0:
        acc_buf[i] = ui + dt * (float)(1.0 / 6.0) * F;
        nxt[i] = ui + dt * 0.5f * F;
        break;
    case 1:
        acc_buf[i] = acc_buf[i] + dt * (float)(1.0 / 3.0) * F;
        nxt[i] = ui + dt * 0.5f * F;
        break;
    case 2:
        acc_buf[i] = acc_buf[i] + dt * (float)(1.0 / 3.0) * F;
        nxt[i] = ui + dt * F;
        break;
    default:
        u[i] = acc_buf[i] + dt * (float)(1.0 / 6.0) * F;
        break;
    }
}

// Coefficients of a step's stages
struct RkCoef {
    double sixth, third, half, one;  // dt / 6, dt / 3, dt / 2, dt
};
RkCoef rk_coef(double dt) { return RkCoef{dt * (1.0 / 6.0), dt * (1.0 / 3.0), dt * 0.5, dt}; }

// nsteps steps on double fields, sliced layout, one cooperative launch (see GridBarrier): a block's slices by its warps (see share_out),
// the first steps of a sweep loaded before its barrier.  A lane adds into two sums in turn, because a dependent FP64 add waits several times the pipe's time for one.
// 161^2 nodes, 49 entries each: 7.6 us a stage (9.0 as launches over CSR rows), 5.0 of them FP64 issue (two instructions an
// entry), 1.55 the barrier.
template <class VT>
__global__ void __launch_bounds__(RUN_THREADS, 1) k_rk4_run(int64_t n, SellView S, const VT *__restrict__ wc, double *u,
                                                           double *acc_buf, double *sa, double *sb,
                                                           const uint8_t *__restrict__ frozen, int64_t nsteps, RkCoef rk,
                                                           GridSync sync)
{
    int64_t s0, s1;
    block_share(S, s0, s1);
    GridBarrier bar{sync};
    bar.check();
    struct Node {
        double si, ui, ai, sum[2];
        bool row, fixed;  // row: this lane updates the node; what it needs is read ahead
    };
    share_out(S, s0, s1);
    if (bar.stopped()) return;
    SliceSweep<4, 1, 1, 1, true, VT> sweep;
    sweep.place(n, S);
    sweep.preload(n, S, wc);
    for (int64_t it = 0; it < 4 * nsteps; it++) {
        const int stage = (int)(it & 3);
        const double *src = stage == 0 ? u : stage == 2 ? sb : sa;
        sweep.run(
            n, S, wc,
            [&](const SellLane &l, bool own) {
                Node v;
                v.row = own && l.i >= 0 && l.h == 0;
                v.si = l.i >= 0 ? src[l.i] : 0.0;
                v.fixed = v.row && frozen && frozen[l.i];
                v.ui = v.row && stage != 3 ? u[l.i] : 0.0;
                v.ai = v.row && stage != 0 ? acc_buf[l.i] : 0.0;
                v.sum[0] = v.sum[1] = 0.0;
                return v;
            },
            [&](int j, double(&x)[1]) { x[0] = src[j]; },
            [&](Node &v, int q, const double(&x)[1], const VT(&w)[1]) { v.sum[q & 1] = fma(x[0] - v.si, (double)w[0], v.sum[q & 1]); },
            [&](const Node &v, double(&p)[1]) { p[0] = v.sum[0] + v.sum[1]; },
            [&](const SellLane &l, const Node &v, const double(&p)[1]) {
                double acc = p[0];
                for (int o = (1 << S.lg_l) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (!v.row) return;
                const double F = v.fixed ? 0.0 : acc;
                if (stage == 3) {
                    u[l.i] = v.ai + rk.sixth * F;
                    return;
                }
                acc_buf[l.i] = stage == 0 ? v.ui + rk.sixth * F : v.ai + rk.third * F;
                (stage == 1 ? sb : sa)[l.i] = v.ui + (stage == 2 ? rk.one : rk.half) * F;
            });
        if (it + 1 == 4 * nsteps) break;
        sweep.preload(n, S, wc);
        if (!bar.wait()) return;
    }
}

// ---------------------------------------------------------------------------------------------
// Launch shapes and the autotuner
// ---------------------------------------------------------------------------------------------
struct Shape {
    int G, UNR;
};

// default shape: enough lanes that UNR entries per lane cover an average stencil
Shape default_shape(const labfm_ctx *ctx, int min_g)
{
    double avg = ctx->n > 0 ? (double)ctx->nnz / (double)ctx->n : 0.0;
    int G = 4;
    while (G < 32 && G * 4 < avg) G *= 2;
    if (G < min_g) G = min_g;
    return Shape{G, 4};
}

unsigned blocks_for(int64_t n, int G) { return (unsigned)((n * G + APPLY_THREADS - 1) / APPLY_THREADS); }

// Coefficients of stage 0 .. 3 of a Burgers run on float fields: of acc (or u), and of nxt
float stage_ca(int stage, double dt) { return (float)dt * (float)(stage == 0 || stage == 3 ? 1.0 / 6.0 : 1.0 / 3.0); }
float stage_cn(int stage, double dt) { return stage == 2 ? (float)dt : (float)dt * 0.5f; }

int log2_of(int G)
{
    int l = 0;
    while ((1 << l) < G) l++;
    return l;
}

template <int NOPS, class FT, class WT>
cudaError_t launch_apply_shape(labfm_ctx *ctx, Shape sh, uint32_t mask, const void *f, void *out, cudaStream_t s)
{
    const unsigned blocks = blocks_for(ctx->n, sh.G);
    auto args = [&](auto kern) {
        kern<<<blocks, APPLY_THREADS, 0, s>>>(ctx->n, ctx->row_ptr.as<int64_t>(), ctx->col.as<int32_t>(),
                                              (const WT *)ctx->w.ptr, (const FT *)f, (FT *)out, mask, log2_of(sh.G));
    };
    switch (sh.UNR) {
    case 2: args(k_apply<NOPS, FT, WT, 2>); break;
    case 8: args(k_apply<NOPS, FT, WT, 8>); break;
    default: args(k_apply<NOPS, FT, WT, 4>); break;
    }
    return cudaGetLastError();
}

template <int CW>
cudaError_t launch_stage_csr(labfm_ctx *ctx, Shape sh, const float *src, float *u, float *acc, float *nxt,
                             const uint8_t *frozen, int stage, double dt, cudaStream_t s)
{
    const unsigned blocks = blocks_for(ctx->n, sh.G);
    const void *wc = ctx->wcomb.ptr;
    const float *wc_lo = CW == CW_DF ? reinterpret_cast<const float *>(ctx->wcomb.as<int2>() + ctx->nnz) : nullptr;
    auto args = [&](auto kern) {
        kern<<<blocks, APPLY_THREADS, 0, s>>>(ctx->n, ctx->row_ptr.as<int64_t>(), ctx->col.as<int32_t>(), wc, wc_lo, src, u,
                                              acc, nxt, frozen, stage, (float)dt, log2_of(sh.G));
    };
    switch (sh.UNR) {
    case 2: args(k_rk4_stage_csr<CW, 2>); break;
    case 8: args(k_rk4_stage_csr<CW, 8>); break;
    default: args(k_rk4_stage_csr<CW, 4>); break;
    }
    return cudaGetLastError();
}

// Time every shape with `run` (which enqueues one launch on ctx->stream) and keep the fastest.
template <class RunFn>
cudaError_t autotune(labfm_ctx *ctx, uint64_t key, int min_g, RunFn run, Shape &best)
{
    auto it = ctx->tuned.find(key);
    if (it != ctx->tuned.end()) {
        best = Shape{(int)(it->second >> 8), (int)(it->second & 0xff)};
        return cudaSuccess;
    }
    best = default_shape(ctx, min_g);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t ce = cudaStreamIsCapturing(ctx->stream, &cap);
    if (ce != cudaSuccess) return ce;
    if (cap != cudaStreamCaptureStatusNone) return cudaSuccess;  // caller is recording a graph: no timing
    if (ctx->n < 4096) {  // too small to time meaningfully
        ctx->tuned[key] = ((uint32_t)best.G << 8) | (uint32_t)best.UNR;
        return cudaSuccess;
    }
    cudaEvent_t e0, e1;
    cudaError_t e = cudaEventCreate(&e0);
    if (e != cudaSuccess) return e;
    e = cudaEventCreate(&e1);
    if (e != cudaSuccess) {
        cudaEventDestroy(e0);
        return e;
    }
    float best_ms = 1e30f;
    const int gs[4] = {4, 8, 16, 32}, us[3] = {2, 4, 8};
    for (int gi = 0; gi < 4 && e == cudaSuccess; gi++) {
        for (int ui = 0; ui < 3 && e == cudaSuccess; ui++) {
            Shape sh{gs[gi], us[ui]};
            if (sh.G < min_g) continue;
            e = run(sh);  // warm-up
            if (e != cudaSuccess) break;
            cudaEventRecord(e0, ctx->stream);
            e = run(sh);
            cudaEventRecord(e1, ctx->stream);
            if (e != cudaSuccess) break;
            e = cudaEventSynchronize(e1);
            float ms = 0.0f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e == cudaSuccess && ms < best_ms) {
                best_ms = ms;
                best = sh;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e == cudaSuccess) ctx->tuned[key] = ((uint32_t)best.G << 8) | (uint32_t)best.UNR;
    return e;
}

// Shapes are tuned per kind of launch, data types and problem class: floor(log2 n) and the mean
// stencil size rounded to an integer, so that rebuilding stencils of the same kind (a moving node
// set, a bench repetition) reuses the choice instead of timing again.
uint64_t tune_key(const labfm_ctx *ctx, int kind, int nops, int fdt, int wdt)
{
    uint64_t lg = 0;
    while (lg < 62 && ((int64_t)1 << (lg + 1)) <= ctx->n) lg++;
    uint64_t deg = ctx->n > 0 ? (uint64_t)((double)ctx->nnz / (double)ctx->n + 0.5) : 0;
    if (deg > 0xffff) deg = 0xffff;
    return (deg << 40) | (lg << 32) | ((uint64_t)kind << 24) | ((uint64_t)nops << 16) | ((uint64_t)fdt << 8) |
           (uint64_t)wdt;
}

template <int NOPS, class FT, class WT>
cudaError_t launch_apply_t(labfm_ctx *ctx, uint32_t mask, const void *f, int fdt, void *out)
{
    const int min_g = NOPS <= 4 ? 4 : 8;  // the reduce-scatter needs G >= NOPS rounded up to 2^k
    Shape sh;
    cudaError_t e = autotune(
        ctx, tune_key(ctx, 1, NOPS, fdt, ctx->wdtype), min_g,
        [&](Shape s) { return launch_apply_shape<NOPS, FT, WT>(ctx, s, mask, f, out, ctx->stream); }, sh);
    if (e != cudaSuccess) return e;
    return launch_apply_shape<NOPS, FT, WT>(ctx, sh, mask, f, out, ctx->stream);
}

template <int NOPS>
cudaError_t launch_apply_n(labfm_ctx *ctx, uint32_t mask, const void *f, int fdt, void *out)
{
    if (ctx->wdtype == LABFM_F64)
        return fdt == LABFM_F64 ? launch_apply_t<NOPS, double, double>(ctx, mask, f, fdt, out)
                                : launch_apply_t<NOPS, float, double>(ctx, mask, f, fdt, out);
    return fdt == LABFM_F64 ? launch_apply_t<NOPS, double, float>(ctx, mask, f, fdt, out)
                            : launch_apply_t<NOPS, float, float>(ctx, mask, f, fdt, out);
}

// Float fields: the launches of nsteps steps on stream s (nsteps = 0: only tunes the launch shape, on ctx->stream)
template <int CW>
cudaError_t enqueue_steps_csr(labfm_ctx *ctx, void *u, double dt, int64_t nsteps, const uint8_t *frozen, cudaStream_t s)
{
    float *uu = (float *)u, *acc = ctx->rk_acc.as<float>(), *sa = ctx->rk_stage_a.as<float>(), *sb = ctx->rk_stage_b.as<float>();
    // tune on stage 0, which reads u and writes only the work buffers
    Shape sh;
    cudaError_t e = autotune(
        ctx, tune_key(ctx, 2, 1, LABFM_F32, ctx->wdtype), 1,
        [&](Shape sp) { return launch_stage_csr<CW>(ctx, sp, uu, uu, acc, sa, frozen, 0, dt, ctx->stream); }, sh);
    if (e != cudaSuccess) return e;
    for (int64_t st = 0; st < nsteps; st++) {
        if ((e = launch_stage_csr<CW>(ctx, sh, uu, uu, acc, sa, frozen, 0, dt, s)) != cudaSuccess) return e;
        if ((e = launch_stage_csr<CW>(ctx, sh, sa, uu, acc, sb, frozen, 1, dt, s)) != cudaSuccess) return e;
        if ((e = launch_stage_csr<CW>(ctx, sh, sb, uu, acc, sa, frozen, 2, dt, s)) != cudaSuccess) return e;
        if ((e = launch_stage_csr<CW>(ctx, sh, sa, uu, acc, nullptr, frozen, 3, dt, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t enqueue_steps_dt(labfm_ctx *ctx, int fmt, void *u, double dt, int64_t nsteps, const uint8_t *frozen,
                             cudaStream_t s)
{
    return fmt == CW_DF ? enqueue_steps_csr<CW_DF>(ctx, u, dt, nsteps, frozen, s)
                        : enqueue_steps_csr<CW_F32>(ctx, u, dt, nsteps, frozen, s);
}

// Steps of a run in one cooperative launch: it holds its SMs until it ends, so that it is kept to tens of milliseconds
// (about 5 ns per thousand entries and stage)
int64_t steps_per_run(const labfm_ctx *ctx) { return std::max<int64_t>(1, (int64_t)1000000000 / (ctx->nnz + 100000)); }

// Double fields: the run as cooperative launches on the context's stream; fn(steps) enqueues one
template <class Fn>
cudaError_t enqueue_runs(const labfm_ctx *ctx, int64_t nsteps, Fn fn)
{
    const int64_t per = steps_per_run(ctx);
    cudaError_t e = cudaSuccess;
    for (int64_t at = 0; at < nsteps && e == cudaSuccess; at += per) e = fn(std::min(per, nsteps - at));
    return e;
}

}  // namespace

cudaError_t launch_apply(labfm_ctx *ctx, uint32_t mask, const void *f, int fdt, void *out)
{
    switch (ctx->n_ops) {
    case 1: return launch_apply_n<1>(ctx, mask, f, fdt, out);
    case 2: return launch_apply_n<2>(ctx, mask, f, fdt, out);
    case 3: return launch_apply_n<3>(ctx, mask, f, fdt, out);
    case 4: return launch_apply_n<4>(ctx, mask, f, fdt, out);
    case 5: return launch_apply_n<5>(ctx, mask, f, fdt, out);
    case 6: return launch_apply_n<6>(ctx, mask, f, fdt, out);
    case 7: return launch_apply_n<7>(ctx, mask, f, fdt, out);
    default: return launch_apply_n<8>(ctx, mask, f, fdt, out);
    }
}

labfm_status run_step(labfm_ctx *ctx, const double *beta, void *u, int fdt, double dt, int64_t nsteps,
                      const uint8_t *frozen)
{
    cudaStream_t s = ctx->stream;
    const int64_t n = ctx->n, nnz = ctx->nnz;
    size_t fsz = fdt == LABFM_F64 ? 8 : 4;
    const int fmt = cw_format(fdt, ctx->wdtype);
    if (cw_sliced(fmt)) {
        labfm_status st = ensure_sell_shape(ctx);
        if (st != LABFM_OK) return st;
    }
    // combined weight, cached while beta, the weights and the storage format are unchanged
    bool same_beta = ctx->wcomb_valid && ctx->wcomb_dtype == fmt;
    for (int d = 0; d < ctx->n_ops && same_beta; d++) same_beta = (ctx->beta_cached[d] == beta[d]);
    if (!same_beta) {
        const size_t bytes = cw_bytes(ctx, fmt);
        LABFM_CUDA_TRY(ctx, ctx->wcomb.reserve(bytes > 0 ? bytes : 8));
        Beta b{};
        for (int d = 0; d < ctx->n_ops; d++) b.v[d] = beta[d];
        const int32_t *cl = ctx->col.as<int32_t>();
        const unsigned blocks = (unsigned)((nnz + 255) / 256);
        if (nnz > 0) {
            switch (fmt) {
            case CW_S64:
                LABFM_CUDA_TRY(ctx, (launch_sell_fill<double, 1>(ctx, ctx->sell, ctx->wcomb.as<double>(),
                                                                Combined<double>{ctx->w.as<double>(), ctx->n_ops, b})));
                break;
            case CW_S32:
                LABFM_CUDA_TRY(ctx, (launch_sell_fill<float, 1>(ctx, ctx->sell, ctx->wcomb.as<float>(),
                                                               Combined<float>{ctx->w.as<float>(), ctx->n_ops, b})));
                break;
            case CW_DF:
                k_combine<double><<<blocks, 256, 0, s>>>(nnz, ctx->n_ops, ctx->w.as<double>(), cl, ctx->wcomb.ptr, fmt, b);
                break;
            default:
                k_combine<float><<<blocks, 256, 0, s>>>(nnz, ctx->n_ops, ctx->w.as<float>(), cl, ctx->wcomb.ptr, fmt, b);
                break;
            }
            LABFM_CUDA_TRY(ctx, cudaGetLastError());
        }
        for (int d = 0; d < ctx->n_ops; d++) ctx->beta_cached[d] = beta[d];
        ctx->wcomb_valid = true;
        ctx->wcomb_dtype = fmt;
    }
    LABFM_CUDA_TRY(ctx, ctx->rk_acc.reserve(fsz * n));
    LABFM_CUDA_TRY(ctx, ctx->rk_stage_a.reserve(fsz * n));
    LABFM_CUDA_TRY(ctx, ctx->rk_stage_b.reserve(fsz * n));

    if (cw_sliced(fmt)) {
        labfm_status st = ensure_sell(ctx);
        if (st != LABFM_OK) return st;
        double *uu = (double *)u, *acc = ctx->rk_acc.as<double>(), *sa = ctx->rk_stage_a.as<double>(), *sb = ctx->rk_stage_b.as<double>();
        const SellView S = sell_view(ctx->sell);
        LABFM_CUDA_TRY(ctx, ensure_sync(ctx));
        cudaError_t e = enqueue_runs(ctx, nsteps, [&](int64_t steps) {
            return fmt == CW_S64 ? launch_run(ctx, S, k_rk4_run<double>, n, S, ctx->wcomb.as<double>(), uu, acc, sa, sb,
                                              frozen, steps, rk_coef(dt), grid_sync(ctx, LABFM_GAVE_UP))
                                 : launch_run(ctx, S, k_rk4_run<float>, n, S, ctx->wcomb.as<float>(), uu, acc, sa, sb,
                                              frozen, steps, rk_coef(dt), grid_sync(ctx, LABFM_GAVE_UP));
        });
        return e == cudaSuccess ? LABFM_OK : cuda_fail(ctx, e, "RK4 run");
    }

    StepGraph &g = ctx->graph;
    const bool same = g.exec && g.u == u && g.frozen == frozen && g.dtype == fdt && g.dt == dt &&
                      g.nsteps == nsteps && g.n == n && g.nnz == nnz && g.wdtype == ctx->wdtype &&
                      g.row_ptr == ctx->row_ptr.ptr && g.col == ctx->col.ptr && g.wc == ctx->wcomb.ptr &&
                      g.acc == ctx->rk_acc.ptr && g.sa == ctx->rk_stage_a.ptr && g.sb == ctx->rk_stage_b.ptr;
    if (!same) {
        g.release();
        if (!ctx->capture_stream) {
            LABFM_CUDA_TRY(ctx, cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking));
        }
        // the capture stream must see the combined weights (enqueued on the context stream)
        LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        cudaGraph_t graph = nullptr;
        // shapes are tuned (on the context stream) before the capture begins
        {
            cudaError_t te = enqueue_steps_dt(ctx, fmt, u, dt, 0, frozen, s);
            if (te != cudaSuccess) return cuda_fail(ctx, te, "RK4 stage tuning");
            // the capture stream must not start before the tuning launches end
            LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        }
        LABFM_CUDA_TRY(ctx, cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = enqueue_steps_dt(ctx, fmt, u, dt, nsteps, frozen, ctx->capture_stream);
        cudaError_t e2 = cudaStreamEndCapture(ctx->capture_stream, &graph);
        if (e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return cuda_fail(ctx, e, "RK4 stage capture");
        }
        LABFM_CUDA_TRY(ctx, e2);
        e = cudaGraphInstantiate(&g.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            g.exec = nullptr;
            return cuda_fail(ctx, e, "cudaGraphInstantiate");
        }
        g.u = u;
        g.frozen = frozen;
        g.dtype = fdt;
        g.dt = dt;
        g.nsteps = nsteps;
        g.n = n;
        g.nnz = nnz;
        g.wdtype = ctx->wdtype;
        g.row_ptr = ctx->row_ptr.ptr;
        g.col = ctx->col.ptr;
        g.wc = ctx->wcomb.ptr;
        g.acc = ctx->rk_acc.ptr;
        g.sa = ctx->rk_stage_a.ptr;
        g.sb = ctx->rk_stage_b.ptr;
    }
    LABFM_CUDA_TRY(ctx, cudaGraphLaunch(g.exec, s));
    return LABFM_OK;
}

}  // namespace labfm

// ---------------------------------------------------------------------------------------------
// Burgers' equation (Sec. 5.3, eq. burgers): du/dt = -(u d/dx + v d/dy) u + sum_{d>=2} beta_d L^d u,
// and the same for v, by the classical RK4 scheme.  The advection coefficients depend on the
// field, so d/dx and d/dy stay separate sums; the linear operators combine into one weight.
// ---------------------------------------------------------------------------------------------
namespace labfm {
namespace {

// Weights of the stages, the third summed in double: (w^0, w^1, sum_{d>=2} beta_d w^d) per entry in CSR order (float
// fields), or in the sliced layout, three runs of 32 per step of a slice (double fields).
template <class WT>
__global__ void k_burg_combine(int64_t nnz, int n_ops, const WT *__restrict__ w, WT *__restrict__ wb, Beta b)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
        const WT *we = w + e * n_ops;
        double s = 0.0;
        for (int d = 2; d < n_ops; d++) s += b.v[d] * (double)we[d];
        wb[3 * e] = we[0];
        wb[3 * e + 1] = we[1];
        wb[3 * e + 2] = (WT)s;
    }
}

template <class WT>
struct BurgersWeights {
    const WT *__restrict__ w;
    int n_ops;
    Beta b;
    __device__ __forceinline__ void operator()(int64_t e, WT *v) const
    {
        const WT *we = w + e * n_ops;
        double s = 0.0;
        for (int d = 2; d < n_ops; d++) s += b.v[d] * (double)we[d];
        v[0] = we[0];
        v[1] = we[1];
        v[2] = (WT)s;
    }
};

// One RK4 stage for the pair (u, v).  With the stage's source fields (su, sv), the advection weights of node i join
// the linear one per entry, c_ji = wl_ji - su_i w^0_ji - sv_i w^1_ji, and
//   F_u = sum_j (su_j - su_i) c_ji,   F_v = sum_j (sv_j - sv_i) c_ji
// (0 on frozen nodes): six FP64 instructions per entry and two sums to combine, where the sums with w^0, w^1 and wl
// apart take eight and six; the FP64 pipe bounds the stage on sets that fit the L2 cache.  Then the stage updates
// of k_rk4_stage_csr for both fields; acc and nxt hold u in [0, n) and v in [n, 2n).  Sums in double unless fields and
// weights are both float.
template <class WT, int UNR>
__global__ void __launch_bounds__(APPLY_THREADS) k_burgers_stage_csr(int64_t n, const int64_t *__restrict__ row_ptr,
                                                                 const int32_t *__restrict__ col,
                                                                 const WT *__restrict__ wb, const float *__restrict__ su,
                                                                 const float *__restrict__ sv, float *__restrict__ u,
                                                                 float *__restrict__ v, float *__restrict__ acc,
                                                                 float *__restrict__ nxt,
                                                                 const uint8_t *__restrict__ frozen, int stage, float ca,
                                                                 float cnx, int lg_g)
{
    using AT = WT;  // float weights: sums in float
    const int G = 1 << lg_g;
    const int lane = threadIdx.x & (G - 1);
    const int64_t i = ((int64_t)blockIdx.x * APPLY_THREADS + threadIdx.x) >> lg_g;
    const bool live = i < n;
    int64_t rs = 0, re = 0;
    AT ui = 0, vi = 0;
    if (live) {
        rs = row_ptr[i];
        re = row_ptr[i + 1];
        ui = (AT)su[i];
        vi = (AT)sv[i];
    }
    int cj[UNR];
    WT w0[UNR], w1[UNR], wl[UNR];
    auto load_batch = [&](int64_t base) {
#pragma unroll
        for (int q = 0; q < UNR; q++) {
            const int64_t e = base + (int64_t)q * G + lane;
            if (e < re) {
                cj[q] = __ldcs(col + e);
                w0[q] = __ldcs(wb + 3 * e);
                w1[q] = __ldcs(wb + 3 * e + 1);
                wl[q] = __ldcs(wb + 3 * e + 2);
            } else {
                cj[q] = -1;
            }
        }
    };
    AT fu = 0, fv = 0;
    for (int64_t base = rs; base < re; base += (int64_t)G * UNR) {
        load_batch(base);
#pragma unroll
        for (int q = 0; q < UNR; q++) {
            if (cj[q] >= 0) {
                const AT c = fma(-vi, (AT)w1[q], fma(-ui, (AT)w0[q], (AT)wl[q]));
                fu = fma((AT)su[cj[q]] - ui, c, fu);
                fv = fma((AT)sv[cj[q]] - vi, c, fv);
            }
        }
    }
    for (int o = G >> 1; o > 0; o >>= 1) {
        fu += __shfl_xor_sync(0xffffffffu, fu, o);
        fv += __shfl_xor_sync(0xffffffffu, fv, o);
    }
    if (!live || lane != 0) return;
    const bool fixed = frozen && frozen[i];
    const float Fu = fixed ? 0.0f : (float)fu;
    const float Fv = fixed ? 0.0f : (float)fv;
    if (stage == 3) {
        u[i] = acc[i] + ca * Fu;
        v[i] = acc[n + i] + ca * Fv;
        return;
    }
    const float u0 = u[i], v0 = v[i];
    acc[i] = (stage == 0 ? u0 : acc[i]) + ca * Fu;
    acc[n + i] = (stage == 0 ? v0 : acc[n + i]) + ca * Fv;
    nxt[i] = u0 + cnx * Fu;
    nxt[n + i] = v0 + cnx * Fv;
}

// The same on double fields (see k_rk4_run).  161^2 nodes: 17.0 us a stage (29.3 as launches), 14 of them FP64 issue.
template <class VT>
__global__ void __launch_bounds__(RUN_THREADS, 1) k_burgers_run(int64_t n, SellView S, const VT *__restrict__ wb, double *u,
                                                               double *v, double *acc, double *sa, double *sb,
                                                               const uint8_t *__restrict__ frozen, int64_t nsteps,
                                                               RkCoef rk, GridSync sync)
{
    int64_t s0, s1;
    block_share(S, s0, s1);
    GridBarrier bar{sync};
    bar.check();
    struct Node {
        double s[2], u0[2], a0[2], f[2];
        bool row, fixed;
    };
    share_out(S, s0, s1);
    if (bar.stopped()) return;
    SliceSweep<2, 3, 2, 2, false, VT> sweep;
    sweep.preload(n, S, wb);
    for (int64_t it = 0; it < 4 * nsteps; it++) {
        const int stage = (int)(it & 3);
        const double *su = stage == 0 ? u : stage == 2 ? sb : sa, *sv = stage == 0 ? v : su + n;
        double *const field[2] = {u, v};
        sweep.run(
            n, S, wb,
            [&](const SellLane &l, bool own) {
                Node b;
                b.row = own && l.i >= 0 && l.h == 0;
                b.fixed = b.row && frozen && frozen[l.i];
                b.s[0] = l.i >= 0 ? su[l.i] : 0.0;
                b.s[1] = l.i >= 0 ? sv[l.i] : 0.0;
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    b.u0[c] = b.row && stage != 3 ? field[c][l.i] : 0.0;
                    b.a0[c] = b.row && stage != 0 ? acc[c * n + l.i] : 0.0;
                    b.f[c] = 0.0;
                }
                return b;
            },
            [&](int j, double(&x)[2]) {
                x[0] = su[j];
                x[1] = sv[j];
            },
            [&](Node &b, int, const double(&x)[2], const VT(&w)[3]) {
                const double c = fma(-b.s[1], (double)w[1], fma(-b.s[0], (double)w[0], (double)w[2]));
                b.f[0] = fma(x[0] - b.s[0], c, b.f[0]);
                b.f[1] = fma(x[1] - b.s[1], c, b.f[1]);
            },
            [&](const Node &b, double(&p)[2]) {
                p[0] = b.f[0];
                p[1] = b.f[1];
            },
            [&](const SellLane &l, const Node &b, const double(&p)[2]) {
                double f[2] = {p[0], p[1]};
                for (int o = (1 << S.lg_l) >> 1; o > 0; o >>= 1) {
                    f[0] += __shfl_xor_sync(0xffffffffu, f[0], o);
                    f[1] += __shfl_xor_sync(0xffffffffu, f[1], o);
                }
                if (!b.row) return;
                double *const nxt = stage == 1 ? sb : sa;
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    const double F = b.fixed ? 0.0 : f[c];
                    if (stage == 3) {
                        field[c][l.i] = b.a0[c] + rk.sixth * F;
                        continue;
                    }
                    acc[c * n + l.i] = stage == 0 ? b.u0[c] + rk.sixth * F : b.a0[c] + rk.third * F;
                    nxt[c * n + l.i] = b.u0[c] + (stage == 2 ? rk.one : rk.half) * F;
                }
            });
        if (it + 1 == 4 * nsteps) break;
        sweep.preload(n, S, wb);
        if (!bar.wait()) return;
    }
}

template <class WT>
cudaError_t launch_burg_stage_csr(labfm_ctx *ctx, Shape sh, const float *su, const float *sv, float *u, float *v,
                                  float *acc, float *nxt, const uint8_t *frozen, int stage, double dt, cudaStream_t s)
{
    const unsigned blocks = blocks_for(ctx->n, sh.G);
    auto args = [&](auto kern) {
        kern<<<blocks, APPLY_THREADS, 0, s>>>(ctx->n, ctx->row_ptr.as<int64_t>(), ctx->col.as<int32_t>(),
                                              ctx->wburg.as<WT>(), su, sv, u, v, acc, nxt, frozen, stage,
                                              stage_ca(stage, dt), stage_cn(stage, dt), log2_of(sh.G));
    };
    switch (sh.UNR) {
    case 2: args(k_burgers_stage_csr<WT, 2>); break;
    case 8: args(k_burgers_stage_csr<WT, 8>); break;
    default: args(k_burgers_stage_csr<WT, 4>); break;
    }
    return cudaGetLastError();
}

template <class WT>
cudaError_t enqueue_burgers_csr(labfm_ctx *ctx, void *u_, void *v_, double dt, int64_t nsteps, const uint8_t *frozen,
                                cudaStream_t s)
{
    const int64_t n = ctx->n;
    float *u = (float *)u_, *v = (float *)v_, *acc = ctx->bu_acc.as<float>();
    float *sa = ctx->bu_stage_a.as<float>(), *sb = ctx->bu_stage_b.as<float>();
    // tune on stage 0, which reads u and v and writes only the work buffers
    Shape sh;
    cudaError_t e = autotune(
        ctx, tune_key(ctx, 3, 2, LABFM_F32, ctx->wdtype), 1,
        [&](Shape sp) { return launch_burg_stage_csr<WT>(ctx, sp, u, v, u, v, acc, sa, frozen, 0, dt, ctx->stream); }, sh);
    if (e != cudaSuccess) return e;
    for (int64_t st = 0; st < nsteps; st++) {
        if ((e = launch_burg_stage_csr<WT>(ctx, sh, u, v, u, v, acc, sa, frozen, 0, dt, s)) != cudaSuccess) return e;
        if ((e = launch_burg_stage_csr<WT>(ctx, sh, sa, sa + n, u, v, acc, sb, frozen, 1, dt, s)) != cudaSuccess) return e;
        if ((e = launch_burg_stage_csr<WT>(ctx, sh, sb, sb + n, u, v, acc, sa, frozen, 2, dt, s)) != cudaSuccess) return e;
        if ((e = launch_burg_stage_csr<WT>(ctx, sh, sa, sa + n, u, v, acc, nullptr, frozen, 3, dt, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t enqueue_burgers_dt(labfm_ctx *ctx, void *u, void *v, double dt, int64_t nsteps, const uint8_t *frozen,
                               cudaStream_t s)
{
    return ctx->wdtype == LABFM_F64 ? enqueue_burgers_csr<double>(ctx, u, v, dt, nsteps, frozen, s)
                                    : enqueue_burgers_csr<float>(ctx, u, v, dt, nsteps, frozen, s);
}

}  // namespace

labfm_status run_step_burgers(labfm_ctx *ctx, const double *beta, void *u, void *v, int fdt, double dt,
                              int64_t nsteps, const uint8_t *frozen)
{
    cudaStream_t s = ctx->stream;
    const int64_t n = ctx->n, nnz = ctx->nnz;
    const size_t fsz = fdt == LABFM_F64 ? 8 : 4, wsz = ctx->wdtype == LABFM_F64 ? 8 : 4;
    const bool sliced = fdt == LABFM_F64;
    if (sliced) {
        labfm_status st = ensure_sell_shape(ctx);
        if (st != LABFM_OK) return st;
    }
    bool same_beta = ctx->wburg_valid && ctx->wburg_sliced == sliced;
    for (int d = 2; d < ctx->n_ops && same_beta; d++) same_beta = (ctx->beta_burg[d] == beta[d]);
    if (!same_beta) {
        const int64_t entries = sliced ? ctx->sell.places : nnz;
        LABFM_CUDA_TRY(ctx, ctx->wburg.reserve(3 * wsz * (size_t)(entries > 0 ? entries : 1)));
        Beta b{};
        for (int d = 2; d < ctx->n_ops; d++) b.v[d] = beta[d];
        if (nnz > 0) {
            auto combine = [&](auto wt) -> cudaError_t {
                using WT = decltype(wt);
                if (sliced)
                    return launch_sell_fill<WT, 3>(ctx, ctx->sell, ctx->wburg.as<WT>(),
                                                   BurgersWeights<WT>{ctx->w.as<WT>(), ctx->n_ops, b});
                k_burg_combine<WT><<<(unsigned)std::min<int64_t>((nnz + 255) / 256, (int64_t)ctx->num_sms * 32), 256, 0, s>>>(
                    nnz, ctx->n_ops, ctx->w.as<WT>(), ctx->wburg.as<WT>(), b);
                return cudaGetLastError();
            };
            LABFM_CUDA_TRY(ctx, ctx->wdtype == LABFM_F64 ? combine(0.0) : combine(0.0f));
        }
        ctx->wburg_sliced = sliced;
        for (int d = 2; d < ctx->n_ops; d++) ctx->beta_burg[d] = beta[d];
        ctx->wburg_valid = true;
    }
    LABFM_CUDA_TRY(ctx, ctx->bu_acc.reserve(2 * fsz * n));
    LABFM_CUDA_TRY(ctx, ctx->bu_stage_a.reserve(2 * fsz * n));
    LABFM_CUDA_TRY(ctx, ctx->bu_stage_b.reserve(2 * fsz * n));

    if (sliced) {
        labfm_status st = ensure_sell(ctx);
        if (st != LABFM_OK) return st;
        double *uu = (double *)u, *vv = (double *)v, *acc = ctx->bu_acc.as<double>();
        double *sa = ctx->bu_stage_a.as<double>(), *sb = ctx->bu_stage_b.as<double>();
        const SellView S = sell_view(ctx->sell);
        LABFM_CUDA_TRY(ctx, ensure_sync(ctx));
        cudaError_t e = enqueue_runs(ctx, nsteps, [&](int64_t steps) {
            return ctx->wdtype == LABFM_F64
                       ? launch_run(ctx, S, k_burgers_run<double>, n, S, ctx->wburg.as<double>(), uu, vv, acc, sa, sb,
                                    frozen, steps, rk_coef(dt), grid_sync(ctx, LABFM_GAVE_UP))
                       : launch_run(ctx, S, k_burgers_run<float>, n, S, ctx->wburg.as<float>(), uu, vv, acc, sa, sb,
                                    frozen, steps, rk_coef(dt), grid_sync(ctx, LABFM_GAVE_UP));
        });
        return e == cudaSuccess ? LABFM_OK : cuda_fail(ctx, e, "Burgers run");
    }

    StepGraph &g = ctx->graph_burgers;
    const bool same = g.exec && g.u == u && g.v == v && g.frozen == frozen && g.dtype == fdt && g.dt == dt &&
                      g.nsteps == nsteps && g.n == n && g.nnz == nnz && g.wdtype == ctx->wdtype &&
                      g.row_ptr == ctx->row_ptr.ptr && g.col == ctx->col.ptr && g.wc == ctx->wburg.ptr &&
                      g.acc == ctx->bu_acc.ptr && g.sa == ctx->bu_stage_a.ptr && g.sb == ctx->bu_stage_b.ptr;
    if (!same) {
        g.release();
        if (!ctx->capture_stream) {
            LABFM_CUDA_TRY(ctx, cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking));
        }
        LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));  // the combined weights, before the capture stream reads them
        {
            cudaError_t te = enqueue_burgers_dt(ctx, u, v, dt, 0, frozen, s);  // tuning only
            if (te != cudaSuccess) return cuda_fail(ctx, te, "Burgers stage tuning");
            LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        }
        cudaGraph_t graph = nullptr;
        LABFM_CUDA_TRY(ctx, cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = enqueue_burgers_dt(ctx, u, v, dt, nsteps, frozen, ctx->capture_stream);
        cudaError_t e2 = cudaStreamEndCapture(ctx->capture_stream, &graph);
        if (e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return cuda_fail(ctx, e, "Burgers stage capture");
        }
        LABFM_CUDA_TRY(ctx, e2);
        e = cudaGraphInstantiate(&g.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            g.exec = nullptr;
            return cuda_fail(ctx, e, "cudaGraphInstantiate");
        }
        g.u = u;
        g.v = v;
        g.frozen = frozen;
        g.dtype = fdt;
        g.dt = dt;
        g.nsteps = nsteps;
        g.n = n;
        g.nnz = nnz;
        g.wdtype = ctx->wdtype;
        g.row_ptr = ctx->row_ptr.ptr;
        g.col = ctx->col.ptr;
        g.wc = ctx->wburg.ptr;
        g.acc = ctx->bu_acc.ptr;
        g.sa = ctx->bu_stage_a.ptr;
        g.sb = ctx->bu_stage_b.ptr;
    }
    LABFM_CUDA_TRY(ctx, cudaGraphLaunch(g.exec, s));
    return LABFM_OK;
}

}  // namespace labfm
