// C ABI of liblabfm: context management, argument checks and dispatch to the kernels.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>

#include "labfm_internal.cuh"

namespace labfm {

cudaError_t DevBuf::reserve(size_t need)
{
    if (need <= bytes && ptr) return cudaSuccess;
    release();
    size_t want = need < 256 ? 256 : need;
    cudaError_t e = cudaMalloc(&ptr, want);
    if (e != cudaSuccess) {
        ptr = nullptr;
        bytes = 0;
        return e;
    }
    bytes = want;
    return cudaSuccess;
}

void DevBuf::release()
{
    if (ptr) cudaFree(ptr);
    ptr = nullptr;
    bytes = 0;
}

void StepGraph::release()
{
    if (exec) cudaGraphExecDestroy(exec);
    exec = nullptr;
    u = nullptr;
    v = nullptr;
    frozen = nullptr;
    dtype = -1;
    nsteps = 0;
}

labfm_status fail(labfm_ctx *ctx, labfm_status st, const std::string &msg)
{
    if (ctx) ctx->err = msg;
    return st;
}

labfm_status cuda_fail(labfm_ctx *ctx, cudaError_t e, const char *where)
{
    char buf[512];
    snprintf(buf, sizeof buf, "CUDA error %d (%s) at %s", (int)e, cudaGetErrorString(e), where);
    return fail(ctx, e == cudaErrorMemoryAllocation ? LABFM_ERR_NOMEM : LABFM_ERR_CUDA, buf);
}

// ---------------------------------------------------------------------------------------------
// Exclusive scan of int32 counts into int64 offsets, out[n] the total.  One launch up to SCAN_ITEMS elements; beyond,
// the sums of the blocks' runs first, then every block adds up the sums before its own (up to SCAN_DIRECT blocks:
// 8 bytes each from L2, less than the launches that scanning them would take; above, they are scanned by a
// recursion) and scans its run.  Two launches for what took four; a small search is mostly launches.
// ---------------------------------------------------------------------------------------------
constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 2 * SCAN_THREADS;
constexpr int64_t SCAN_DIRECT = 4096;

// Sum over the block, on every thread.
__device__ __forceinline__ int64_t scan_block_sum(int64_t v, int64_t *sh)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = sh[threadIdx.x & 31];  // SCAN_THREADS / 32 = 32 warps
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();  // sh is free again
    return v;
}

template <class Tin>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_sums(const Tin *__restrict__ in, int64_t n, int64_t *__restrict__ sums)
{
    __shared__ int64_t sh[32];
    const int64_t g = (int64_t)blockIdx.x * SCAN_ITEMS + threadIdx.x;
    int64_t v = g < n ? (int64_t)in[g] : 0;
    if (g + SCAN_THREADS < n) v += (int64_t)in[g + SCAN_THREADS];
    v = scan_block_sum(v, sh);
    if (threadIdx.x == 0) sums[blockIdx.x] = v;
}

// sums: the sums of the blocks' runs, or with `scanned` their exclusive scan; null for a single block
template <class Tin>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_apply(const Tin *__restrict__ in, int64_t *__restrict__ out, int64_t n,
                                                             const int64_t *__restrict__ sums, int scanned,
                                                             unsigned long long *__restrict__ largest)
{
    __shared__ int64_t sh[32];
    __shared__ unsigned sh_max[32];
    int64_t before = 0;  // the sum of all earlier blocks' runs
    if (sums && scanned) {
        before = sums[blockIdx.x];
    } else if (sums) {
        for (int64_t b = threadIdx.x; b < blockIdx.x; b += SCAN_THREADS) before += sums[b];
        before = scan_block_sum(before, sh);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t g = (int64_t)blockIdx.x * SCAN_ITEMS + 2 * threadIdx.x;
    const int64_t a = g < n ? (int64_t)in[g] : 0, b = g + 1 < n ? (int64_t)in[g + 1] : 0;
    int64_t v = a + b;  // inclusive scan of the threads' pairs
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t w = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += w;
    }
    if (lane == 31) sh[warp] = v;
    if (largest) sh_max[warp] = __reduce_max_sync(0xffffffffu, (unsigned)max(a, b));
    __syncthreads();
    int64_t ws = lane < warp ? sh[lane] : 0;
    for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
    const int64_t at = before + ws + v - (a + b);
    if (g < n) out[g] = at;
    if (g + 1 < n) out[g + 1] = at + a;
    if (g < n && g + 2 >= n) out[n] = at + a + b;  // the thread of the last element
    if (largest && warp == 0) {
        const unsigned most = __reduce_max_sync(0xffffffffu, sh_max[lane]);
        if (lane == 0) atomicMax(largest, (unsigned long long)most);
    }
}

__global__ void k_scan_empty(int64_t *out) { out[0] = 0; }

template <class Tin>
static cudaError_t scan_rec(const Tin *in, int64_t *out, int64_t n, int64_t *tmp, cudaStream_t s, unsigned long long *largest)
{
    const int64_t nb = (n + SCAN_ITEMS - 1) / SCAN_ITEMS;
    int64_t *sums = nullptr;
    if (nb > 1) {
        sums = tmp;
        k_scan_sums<Tin><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, sums);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (nb > SCAN_DIRECT) {
            int64_t *scanned = tmp + nb;  // nb + 1 elements
            if ((e = scan_rec<int64_t>(sums, scanned, nb, tmp + 2 * nb + 1, s, nullptr)) != cudaSuccess) return e;
            sums = scanned;
        }
    }
    k_scan_apply<Tin><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, out, n, sums, nb > SCAN_DIRECT ? 1 : 0, largest);
    return cudaGetLastError();
}

size_t scan_workspace_elems(int64_t n)
{
    size_t tot = 0;
    while (true) {
        int64_t nb = (n + SCAN_ITEMS - 1) / SCAN_ITEMS;
        if (nb <= 1) break;
        tot += 2 * nb + 1;
        n = nb;
    }
    return tot + 16;
}

cudaError_t exclusive_scan_i32_to_i64_ws(const int32_t *in, int64_t *out, int64_t n, int64_t *tmp, size_t tmp_elems,
                                         cudaStream_t s, unsigned long long *largest)
{
    if (scan_workspace_elems(n) > tmp_elems) return cudaErrorInvalidValue;
    if (n > 0) return scan_rec<int32_t>(in, out, n, tmp, s, largest);
    k_scan_empty<<<1, 1, 0, s>>>(out);
    return cudaGetLastError();
}

cudaError_t exclusive_scan_i32_to_i64(const int32_t *in, int64_t *out, int64_t n, DevBuf &tmp, cudaStream_t s,
                                      unsigned long long *largest)
{
    const size_t elems = scan_workspace_elems(n);
    cudaError_t e = tmp.reserve(elems * sizeof(int64_t));
    return e == cudaSuccess ? exclusive_scan_i32_to_i64_ws(in, out, n, tmp.as<int64_t>(), elems, s, largest) : e;
}

}  // namespace labfm

using namespace labfm;

extern "C" {

labfm_status labfm_create(labfm_ctx **out, int device, void *stream)
{
    if (!out) return LABFM_ERR_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return LABFM_ERR_CUDA;
    if (cudaSetDevice(device) != cudaSuccess) return LABFM_ERR_CUDA;
    labfm_ctx *ctx = new (std::nothrow) labfm_ctx();
    if (!ctx) return LABFM_ERR_NOMEM;
    ctx->device = device;
    ctx->stream = (cudaStream_t)stream;
    cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, device);
    ctx->run_blocks = ctx->num_sms;
    if (cudaMallocHost(&ctx->host_small, 1024) != cudaSuccess) {  // status words read back by the calls
        delete ctx;
        return LABFM_ERR_NOMEM;
    }
    memset(ctx->host_small, 0, 1024);
    *out = ctx;
    return LABFM_OK;
}

void labfm_destroy(labfm_ctx *ctx)
{
    if (!ctx) return;
    cudaSetDevice(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    DevBuf *bufs[] = {&ctx->node_xy, &ctx->node_h, &ctx->row_ptr, &ctx->col, &ctx->cell_of, &ctx->cell_count, &ctx->cell_start,
                      &ctx->cell_nodes, &ctx->counts, &ctx->scan_tmp, &ctx->misc, &ctx->w,
                      &ctx->status_tmp, &ctx->wtilde, &ctx->mscratch, &ctx->mrecs, &ctx->mwstore, &ctx->mfallback, &ctx->wcomb, &ctx->rk_acc,
                      &ctx->rk_stage_a, &ctx->rk_stage_b, &ctx->wburg, &ctx->bu_acc, &ctx->bu_stage_a,
                      &ctx->bu_stage_b, &ctx->sol_w, &ctx->sol_vec, &ctx->sol_part, &ctx->sol_gmap, &ctx->sync_buf};
    for (DevBuf *b : bufs) b->release();
    ctx->sell.release();
    ctx->sell_ghost.release();
    ctx->graph.release();
    ctx->graph_burgers.release();
    if (ctx->capture_stream) cudaStreamDestroy(ctx->capture_stream);
    if (ctx->host_small) cudaFreeHost(ctx->host_small);
    delete ctx;
}

const char *labfm_last_error(const labfm_ctx *ctx) { return ctx ? ctx->err.c_str() : "null context"; }

labfm_status labfm_set_stream(labfm_ctx *ctx, void *stream)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->stream = (cudaStream_t)stream;
    ctx->run_blocks = ctx->num_sms;
    ctx->graph.release();
    ctx->graph_burgers.release();
    return LABFM_OK;
}

labfm_status labfm_build_neighbours(labfm_ctx *ctx, int64_t n, const double *xy, const double *h, int periodic,
                                    const double box_lo[2], const double box_hi[2], int64_t *nnz_out)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->err.clear();
    if (n < 1 || n >= ((int64_t)1 << 31)) return fail(ctx, LABFM_ERR_ARG, "n must be in [1, 2^31)");
    if (!xy || !h || !box_lo || !box_hi || !nnz_out) return fail(ctx, LABFM_ERR_ARG, "null pointer argument");
    for (int d = 0; d < 2; d++)
        if (!std::isfinite(box_lo[d]) || !std::isfinite(box_hi[d]) || !(box_hi[d] > box_lo[d]))
            return fail(ctx, LABFM_ERR_ARG, "box must be finite with box_hi > box_lo");
    if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, LABFM_ERR_CUDA, "cudaSetDevice failed");
    ctx->have_weights = false;
    ctx->wcomb_valid = false;
    ctx->sell.shaped = ctx->sell.valid = false;
    const labfm_status st = run_neighbours(ctx, n, xy, h, periodic ? 1 : 0, box_lo, box_hi, nnz_out);
    const labfm_status rs = run_gave_up(ctx);  // (every run has ended: the search waited for the stream)
    if (rs != LABFM_OK) ctx->n = 0;            // its positions may come from that run
    return rs != LABFM_OK ? rs : st;
}

labfm_status labfm_get_neighbours(labfm_ctx *ctx, const int64_t **row_ptr, const int32_t **col, int64_t *n,
                                  int64_t *nnz)
{
    if (!ctx) return LABFM_ERR_ARG;
    if (ctx->n == 0) return fail(ctx, LABFM_ERR_STATE, "no stencils built");
    if (row_ptr) *row_ptr = ctx->row_ptr.as<int64_t>();
    if (col) *col = ctx->col.as<int32_t>();
    if (n) *n = ctx->n;
    if (nnz) *nnz = ctx->nnz;
    return LABFM_OK;
}

labfm_status labfm_build_weights(labfm_ctx *ctx, const int8_t *order, int uniform_order, int rbf, int n_ops,
                                 const double *C, int precision, int weight_dtype, int32_t *node_status,
                                 int64_t *n_bad_out)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->err.clear();
    if (ctx->n == 0) return fail(ctx, LABFM_ERR_STATE, "labfm_build_neighbours must come first");
    if (!order && (uniform_order < 1 || uniform_order > LABFM_MAX_ORDER))
        return fail(ctx, LABFM_ERR_ARG, "uniform_order must be in 1..8");
    {
        int base = rbf & LABFM_RBF_MASK, form = rbf & ~LABFM_RBF_MASK;
        if (base < LABFM_RBF_WENDLAND_C2 || base > LABFM_RBF_GAUSSIAN || (form & ~LABFM_ABF_DW0_ONLY))
            return fail(ctx, LABFM_ERR_ARG, "unknown rbf");
    }
    if (n_ops < 1 || n_ops > LABFM_MAX_OPS) return fail(ctx, LABFM_ERR_ARG, "n_ops must be in 1..8");
    if (!C) return fail(ctx, LABFM_ERR_ARG, "C is null");
    for (int t = 0; t < n_ops * LABFM_PMAX; t++)
        if (!std::isfinite(C[t])) return fail(ctx, LABFM_ERR_ARG, "C has a non-finite entry");
    {
        int base = precision & 0xff, forced = (precision >> 8) & 0xf, rest = precision >> 12;
        bool ok = rest == 0 && (base == LABFM_PREC_FP64
                                    ? forced == 0
                                    : ((base == LABFM_PREC_MIXED || base == LABFM_PREC_MIXED_TC) && forced <= 5));
        if (!ok) return fail(ctx, LABFM_ERR_ARG, "unknown precision");
    }
    if (weight_dtype != LABFM_F64 && weight_dtype != LABFM_F32) return fail(ctx, LABFM_ERR_ARG, "bad weight_dtype");
    if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, LABFM_ERR_CUDA, "cudaSetDevice failed");
    ctx->have_weights = false;
    ctx->wcomb_valid = false;
    ctx->wburg_valid = false;
    labfm_status st =
        run_build(ctx, order, uniform_order, rbf, n_ops, C, precision, weight_dtype, node_status, n_bad_out);
    if (const labfm_status rs = run_gave_up(ctx)) return rs;
    if (st == LABFM_OK || st == LABFM_ERR_SINGULAR) {
        ctx->have_weights = true;
        ctx->n_ops = n_ops;
        ctx->wdtype = weight_dtype;
        // operators 0 and 1 are d/dx and d/dy when their targets are the unit vectors of the
        // first two elements of D (Sec. 2): what labfm_step_burgers needs
        bool g = n_ops >= 2;
        for (int e = 0; e < LABFM_PMAX && g; e++)
            g = C[e] == (e == 0 ? 1.0 : 0.0) && C[LABFM_PMAX + e] == (e == 1 ? 1.0 : 0.0);
        ctx->grad01 = g;
    }
    return st;
}

labfm_status labfm_get_build_info(labfm_ctx *ctx, labfm_build_info *info)
{
    if (!ctx || !info) return LABFM_ERR_ARG;
    if (!ctx->have_weights) return fail(ctx, LABFM_ERR_STATE, "no weights built");
    for (int t = 0; t < 8; t++) info->refine_steps[t] = ctx->info_ref_hist[t];
    info->fp64_rebuilt = ctx->info_fp64_rebuilt;
    for (int k = 0; k <= LABFM_MAX_ORDER; k++) {
        info->fp64_group_threads[k] = ctx->info_group[k];
        info->mixed_inv_threads_per_row[k] = ctx->info_inv_tpr[k];
    }
    return LABFM_OK;
}

labfm_status labfm_get_weights(labfm_ctx *ctx, const void **w, int *dtype, int *n_ops)
{
    if (!ctx) return LABFM_ERR_ARG;
    if (!ctx->have_weights) return fail(ctx, LABFM_ERR_STATE, "no weights built");
    if (w) *w = ctx->w.ptr;
    if (dtype) *dtype = ctx->wdtype;
    if (n_ops) *n_ops = ctx->n_ops;
    return LABFM_OK;
}

labfm_status labfm_apply(labfm_ctx *ctx, uint32_t op_mask, const void *f, int field_dtype, void *out)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->err.clear();
    if (!ctx->have_weights) return fail(ctx, LABFM_ERR_STATE, "labfm_build_weights must come first");
    if (const labfm_status rs = run_gave_up(ctx)) return rs;
    if (!f || !out) return fail(ctx, LABFM_ERR_ARG, "null field or output");
    if (field_dtype != LABFM_F64 && field_dtype != LABFM_F32) return fail(ctx, LABFM_ERR_ARG, "bad field_dtype");
    if (op_mask == 0 || (op_mask >> ctx->n_ops) != 0) return fail(ctx, LABFM_ERR_ARG, "op_mask selects no or unknown operators");
    cudaError_t e = launch_apply(ctx, op_mask, f, field_dtype, out);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "labfm_apply launch");
    return LABFM_OK;
}

labfm_status labfm_step(labfm_ctx *ctx, const double *beta, void *u, int field_dtype, double dt, int64_t nsteps,
                        const uint8_t *frozen)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->err.clear();
    if (!ctx->have_weights) return fail(ctx, LABFM_ERR_STATE, "labfm_build_weights must come first");
    if (const labfm_status rs = run_gave_up(ctx)) return rs;
    if (!beta || !u) return fail(ctx, LABFM_ERR_ARG, "null beta or u");
    if (field_dtype != LABFM_F64 && field_dtype != LABFM_F32) return fail(ctx, LABFM_ERR_ARG, "bad field_dtype");
    if (!std::isfinite(dt) || nsteps < 0) return fail(ctx, LABFM_ERR_ARG, "dt must be finite and nsteps >= 0");
    for (int d = 0; d < ctx->n_ops; d++)
        if (!std::isfinite(beta[d])) return fail(ctx, LABFM_ERR_ARG, "beta has a non-finite entry");
    if (nsteps == 0) return LABFM_OK;
    return run_step(ctx, beta, u, field_dtype, dt, nsteps, frozen);
}

labfm_status labfm_solve(labfm_ctx *ctx, int op, const double *f, double *phi, const uint8_t *dirichlet, double tol,
                         int max_iter, int *iters_out, double *resid_out)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->err.clear();
    if (!ctx->have_weights) return fail(ctx, LABFM_ERR_STATE, "labfm_build_weights must come first");
    if (const labfm_status rs = run_gave_up(ctx)) return rs;
    if (op < 0 || op >= ctx->n_ops) return fail(ctx, LABFM_ERR_ARG, "op must index a built operator");
    if (!f || !phi) return fail(ctx, LABFM_ERR_ARG, "null f or phi");
    if ((const void *)f == (const void *)phi) return fail(ctx, LABFM_ERR_ARG, "f and phi must be distinct buffers");
    if (!(tol > 0.0) || !std::isfinite(tol) || max_iter < 1) return fail(ctx, LABFM_ERR_ARG, "need tol > 0 and max_iter >= 1");
    return run_solve(ctx, op, f, phi, dirichlet, SolveNeumann{}, tol, max_iter, iters_out, resid_out);
}

labfm_status labfm_solve_neumann(labfm_ctx *ctx, int op, const double *f, double *phi, const uint8_t *dirichlet,
                                 int64_t n_ghost, const int64_t *ghost, const int64_t *parent, const double *normal,
                                 int op_x, int op_y, double tol, int max_iter, int *iters_out, double *resid_out)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->err.clear();
    if (!ctx->have_weights) return fail(ctx, LABFM_ERR_STATE, "labfm_build_weights must come first");
    if (const labfm_status rs = run_gave_up(ctx)) return rs;
    if (op < 0 || op >= ctx->n_ops) return fail(ctx, LABFM_ERR_ARG, "op must index a built operator");
    if (!f || !phi) return fail(ctx, LABFM_ERR_ARG, "null f or phi");
    if ((const void *)f == (const void *)phi) return fail(ctx, LABFM_ERR_ARG, "f and phi must be distinct buffers");
    if (!(tol > 0.0) || !std::isfinite(tol) || max_iter < 1) return fail(ctx, LABFM_ERR_ARG, "need tol > 0 and max_iter >= 1");
    if (n_ghost < 0 || n_ghost > ctx->n) return fail(ctx, LABFM_ERR_ARG, "need 0 <= n_ghost <= n");
    SolveNeumann nm;
    if (n_ghost > 0) {
        if (!ghost || !parent || !normal) return fail(ctx, LABFM_ERR_ARG, "null ghost, parent or normal");
        if (op_x < 0 || op_x >= ctx->n_ops || op_y < 0 || op_y >= ctx->n_ops)
            return fail(ctx, LABFM_ERR_ARG, "op_x and op_y must index built operators");
        nm.n_ghost = n_ghost;
        nm.ghost = ghost;
        nm.parent = parent;
        nm.normal = normal;
        nm.op_x = op_x;
        nm.op_y = op_y;
    }
    return run_solve(ctx, op, f, phi, dirichlet, nm, tol, max_iter, iters_out, resid_out);
}

labfm_status labfm_step_burgers(labfm_ctx *ctx, const double *beta, void *u, void *v, int field_dtype, double dt,
                                int64_t nsteps, const uint8_t *frozen)
{
    if (!ctx) return LABFM_ERR_ARG;
    ctx->err.clear();
    if (!ctx->have_weights) return fail(ctx, LABFM_ERR_STATE, "labfm_build_weights must come first");
    if (const labfm_status rs = run_gave_up(ctx)) return rs;
    if (!ctx->grad01) return fail(ctx, LABFM_ERR_ARG, "operators 0 and 1 of the weights must be d/dx and d/dy");
    if (!beta || !u || !v) return fail(ctx, LABFM_ERR_ARG, "null beta, u or v");
    if (u == v) return fail(ctx, LABFM_ERR_ARG, "u and v must be distinct buffers");
    if (field_dtype != LABFM_F64 && field_dtype != LABFM_F32) return fail(ctx, LABFM_ERR_ARG, "bad field_dtype");
    if (!std::isfinite(dt) || nsteps < 0) return fail(ctx, LABFM_ERR_ARG, "dt must be finite and nsteps >= 0");
    for (int d = 2; d < ctx->n_ops; d++)
        if (!std::isfinite(beta[d])) return fail(ctx, LABFM_ERR_ARG, "beta has a non-finite entry");
    if (nsteps == 0) return LABFM_OK;
    return run_step_burgers(ctx, beta, u, v, field_dtype, dt, nsteps, frozen);
}

}  // extern "C"
