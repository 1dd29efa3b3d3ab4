// The sliced layout of the stencils that the FP64 products read (RK4 and Burgers stages on double fields, implicit
// solves): a slice is 32 / L consecutive nodes, L lanes to a node, and step k of a slice holds entry k L + h of the
// node of lane (node, h) at place (off[slice] + k) 32 + lane, -1 where the node has no such entry.
//
// A warp then reads indices and weights of a step as one contiguous segment however few lanes a node has.  Read from
// CSR rows the same warp needs 8 lanes a node or so to use the cache lines it touches, and pays for them in FP64
// instructions that most lanes do nothing in: the sums over the lanes and the updates of a node take the FP64 pipe
// (2 lanes per SM and clock) as long as an entry of all 32.  With one or two lanes a node they are a few percent.
#include <algorithm>

#include "sell_fill.cuh"

namespace labfm {
namespace {

constexpr int SELL_THREADS = 256;

// the stencil of row i: its own, or its parent's for a Neumann ghost row
__device__ __forceinline__ int64_t stencil_of(int64_t i, const int32_t *gmap, const int64_t *parent)
{
    if (!gmap) return i;
    const int g = gmap[i];
    return g >= 0 ? parent[g] : i;
}

// steps of every slice (a warp per slice)
__global__ void __launch_bounds__(SELL_THREADS) k_sell_steps(int64_t n, int lg_l, int64_t n_slices,
                                                            const int64_t *__restrict__ row_ptr,
                                                            const int32_t *__restrict__ gmap,
                                                            const int64_t *__restrict__ parent,
                                                            int32_t *__restrict__ steps)
{
    const int lane = threadIdx.x & 31;
    const int64_t slice = (int64_t)blockIdx.x * (SELL_THREADS / 32) + (threadIdx.x >> 5);
    if (slice >= n_slices) return;
    const int64_t i = slice * (32 >> lg_l) + (lane >> lg_l);
    int len = 0;
    if (i < n) {
        const int64_t r = stencil_of(i, gmap, parent);
        len = (int)(row_ptr[r + 1] - row_ptr[r]);
    }
    const int most = __reduce_max_sync(0xffffffffu, len);
    if (lane == 0) steps[slice] = (most + (1 << lg_l) - 1) >> lg_l;
}

// columns and shares of a layout with ghost rows (a warp per slice)
__global__ void __launch_bounds__(SELL_THREADS) k_sell_cols(int64_t n, int lg_l, int64_t n_slices,
                                                           const int64_t *__restrict__ row_ptr,
                                                           const int32_t *__restrict__ col,
                                                           const int32_t *__restrict__ gmap,
                                                           const int64_t *__restrict__ parent,
                                                           const int64_t *__restrict__ off, int32_t *__restrict__ scol,
                                                           int64_t *__restrict__ share, int blocks)
{
    const int lane = threadIdx.x & 31, h = lane & ((1 << lg_l) - 1);
    const int64_t slice = (int64_t)blockIdx.x * (SELL_THREADS / 32) + (threadIdx.x >> 5);
    if (slice >= n_slices) return;
    const int64_t i = slice * (32 >> lg_l) + (lane >> lg_l);
    int64_t rs = 0, re = 0;
    if (i < n) {
        const int64_t r = stencil_of(i, gmap, parent);
        rs = row_ptr[r];
        re = row_ptr[r + 1];
    }
    const int64_t at = off[slice], steps = off[slice + 1] - at;
    if (lane == 0 && share) note_shares(slice, n_slices, off, share, blocks);
    for (int64_t k = 0; k < steps; k++) {
        const int64_t e = rs + (k << lg_l) + h;
        scol[(at + k) * 32 + lane] = e < re ? col[e] : -1;
    }
}

}  // namespace

// Lanes per node, as the power of two with the least cost of a sweep of the busiest block.  It is the larger of two, in cycles:
// 16 per FP64 instruction, two per entry of a lane, about four for the node and two per combining step; and 210 per
// place of the longest warp for its loads (see share_out: whole slices, or cut ones where those are more uneven); of
// the same size they add up, about as the fourth root of the sum of fourth powers.  One lane for large sets, two at 129^2 and
// 161^2 nodes, sixteen at 41^2.  Over 45 sizes of heat, Burgers, solver and order-8 runs between 41^2 and 900^2 the
// choice is within 0.3 % of the best lane count on average and 4 % at worst.
static int sell_lanes_log2(int64_t n, int64_t nnz, int num_sms)
{
    const int64_t deg = n > 0 ? (nnz + n - 1) / n : 0;
    int best = 0;
    double least = 0.0;
    for (int lg = 0; lg <= 4; lg++) {
        const int64_t slices = ((n << lg) + 31) / 32, most = (slices + num_sms - 1) / num_sms;
        const int64_t steps = (deg + (1 << lg) - 1) >> lg, whole = (most + RUN_WARPS - 1) / RUN_WARPS * (steps + SLICE_COST);
        const int64_t cut = most * (steps + SLICE_COST) / RUN_WARPS + CUT_COST;
        const double issue = 16.0 * (double)(most * (2 * steps + 2 * lg + 4)), loads = 210.0 * (double)std::min(whole, cut);
        const double cost = issue * issue * issue * issue + loads * loads * loads * loads;
        if (lg == 0 || cost < least) {
            least = cost;
            best = lg;
        }
    }
    return best;
}

// Blocks get equal numbers of places where slices differ in length (order 6 on 200^2 nodes graded towards walls: 14.9 -> 11.3 us a
// stage), but equal numbers of slices where no row is half as long again as the mean: a few shorter ones at the box's
// edge would otherwise make a block with one slice more than warps (193^2: 10.5 us a stage, 12.5 by places).
static bool even_rows(const labfm_ctx *ctx) { return 2 * ctx->longest * ctx->n <= 3 * ctx->nnz; }

// The layout's shape: lanes per node and the places of the slices.  The longest row, which the search has counted, bounds
// the places of ordinary sets, so that their number need not be waited for.
static labfm_status shape_sell(labfm_ctx *ctx, Sell &L, const int32_t *gmap, const int64_t *parent)
{
    cudaStream_t s = ctx->stream;
    const int64_t n = ctx->n, most_places = 2 * ctx->nnz + 64 * n;
    L.shaped = L.valid = false;
    L.lg_l = sell_lanes_log2(n, ctx->nnz, ctx->num_sms);
    while (true) {
        const int64_t per = 32 >> L.lg_l;
        L.n_slices = (n + per - 1) / per;
        LABFM_CUDA_TRY(ctx, L.steps.reserve(sizeof(int32_t) * L.n_slices));
        LABFM_CUDA_TRY(ctx, L.off.reserve(sizeof(int64_t) * (L.n_slices + 1)));
        k_sell_steps<<<(unsigned)((L.n_slices + SELL_THREADS / 32 - 1) / (SELL_THREADS / 32)), SELL_THREADS, 0, s>>>(
            n, L.lg_l, L.n_slices, ctx->row_ptr.as<int64_t>(), gmap, parent, L.steps.as<int32_t>());
        LABFM_CUDA_TRY(ctx, cudaGetLastError());
        LABFM_CUDA_TRY(ctx, exclusive_scan_i32_to_i64(L.steps.as<int32_t>(), L.off.as<int64_t>(), L.n_slices, ctx->scan_tmp, s));
        L.places = 32 * L.n_slices * ((ctx->longest + (1 << L.lg_l) - 1) >> L.lg_l);
        if (L.places <= most_places) break;
        int64_t *total = (int64_t *)ctx->host_small;
        LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(total, L.off.as<int64_t>() + L.n_slices, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        L.places = 32 * *total;
        // a set whose neighbouring nodes differ too much in stencil size (a slice is as long as its largest one):
        // a warp per node, at most 31 places left empty each
        if (L.lg_l == 5 || L.places <= most_places) break;
        L.lg_l = 5;
    }
    L.blocks = (int)std::min<int64_t>(L.n_slices, ctx->num_sms);
    L.even = even_rows(ctx) && L.blocks <= 250;
    const int64_t rounds = ((L.n_slices + L.blocks - 1) / L.blocks + RUN_WARPS - 1) / RUN_WARPS;
    L.whole = L.even && rounds * (((ctx->longest + (1 << L.lg_l) - 1) >> L.lg_l) + SLICE_COST) <= CUT_COST;
    LABFM_CUDA_TRY(ctx, L.col.reserve(sizeof(int32_t) * (L.places > 0 ? L.places : 1)));
    LABFM_CUDA_TRY(ctx, L.share.reserve(sizeof(int64_t) * (L.blocks + 1)));
    L.shaped = true;
    return LABFM_OK;
}

labfm_status build_sell(labfm_ctx *ctx, Sell &L, const int32_t *gmap, const int64_t *parent)
{
    const labfm_status st = shape_sell(ctx, L, gmap, parent);
    if (st != LABFM_OK) return st;
    k_sell_cols<<<(unsigned)((L.n_slices + SELL_THREADS / 32 - 1) / (SELL_THREADS / 32)), SELL_THREADS, 0, ctx->stream>>>(
        ctx->n, L.lg_l, L.n_slices, ctx->row_ptr.as<int64_t>(), ctx->col.as<int32_t>(), gmap, parent, L.off.as<int64_t>(),
        L.col.as<int32_t>(), L.even ? nullptr : L.share.as<int64_t>(), L.blocks);
    LABFM_CUDA_TRY(ctx, cudaGetLastError());
    L.valid = true;
    return LABFM_OK;
}

labfm_status ensure_sell_shape(labfm_ctx *ctx)
{
    return ctx->sell.shaped ? LABFM_OK : shape_sell(ctx, ctx->sell, nullptr, nullptr);
}

struct ColumnsOnly {};

labfm_status ensure_sell(labfm_ctx *ctx)
{
    const labfm_status st = ensure_sell_shape(ctx);
    if (st != LABFM_OK || ctx->sell.valid) return st;
    LABFM_CUDA_TRY(ctx, (launch_sell_fill<int32_t, 0>(ctx, ctx->sell, (int32_t *)nullptr, ColumnsOnly{})));
    return LABFM_OK;
}

}  // namespace labfm
