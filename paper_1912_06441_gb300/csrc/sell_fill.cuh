// Values of the stencils' entries into the sliced layout (see sell.cu), and with them, on the first use of the layout,
// its columns and the blocks' shares.
//
// A block per slice: its rows lie one behind another in CSR order, so that a warp per row reads indices and weights as
// contiguous segments, keeps what it makes of them in shared memory, and the block writes the slice's steps from there,
// 32 places each.  (A lane per place reading CSR entries itself, a row apart from the next lane's, and the columns in a
// launch of their own took 182 and 35 us at 512^2 nodes, order 8, four operators; a step after a rebuild took 570 us
// there and takes 488, 508 as launches over CSR rows.  With 128 threads a block 516, with the loop over a row
// unrolled 549.)
#pragma once

#include "labfm_internal.cuh"

namespace labfm {

constexpr int FILL_THREADS = 256;
constexpr int FILL_SMEM = 96 * 1024;  // slices that need more are read place by place

struct SellFill {
    int64_t n, n_slices;
    int lg_l, cap;  // cap: entries that the block's shared memory holds
    const int64_t *off, *row_ptr;
    const int32_t *col;
    int32_t *scol;   // null: the columns are there
    int64_t *share;  // null: equal numbers of slices
    int blocks;
};

// Where share b of the blocks begins: at the first slice at or behind place b / blocks of all (slice s: those that are s + 1).
__device__ __forceinline__ void note_shares(int64_t slice, int64_t n_slices, const int64_t *off, int64_t *share, int blocks)
{
    const int64_t total = off[n_slices] + SLICE_COST * n_slices;
    const int64_t p0 = off[slice] + SLICE_COST * slice, p1 = off[slice + 1] + SLICE_COST * (slice + 1);
    if (slice == 0) share[0] = 0;
    for (int64_t b = p0 * blocks / total; b <= blocks && total * b / blocks <= p1; b++)
        if (total * b / blocks > p0) share[b] = slice + 1;
}

// fn(e, v): the NV values of entry e in CSR order
template <class VT, int NV, class Fn>
__global__ void __launch_bounds__(FILL_THREADS) k_sell_fill(const __grid_constant__ SellFill F, VT *__restrict__ out,
                                                            const __grid_constant__ Fn fn)
{
    extern __shared__ __align__(16) unsigned char fill_smem[];
    VT *const sv = reinterpret_cast<VT *>(fill_smem);                          // [NV][cap]
    int32_t *const sc = reinterpret_cast<int32_t *>(sv + (size_t)NV * F.cap);  // [cap]
    __shared__ int64_t s_row[32];             // where each row begins in CSR order
    __shared__ int s_len[32], s_at[33];       // its entries, and its place in sv and sc
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t slice = blockIdx.x;
    const int per = 32 >> F.lg_l;
    if (warp == 0) {
        const int64_t i = slice * per + lane;
        int64_t rs = 0;
        int len = 0;
        if (lane < per && i < F.n) {
            rs = F.row_ptr[i];
            len = (int)(F.row_ptr[i + 1] - rs);
        }
        const int room = min(len | 1, 1 << 24);  // odd: rows of equal length begin on different banks (bounded: 32 of them fit an int)
        int end = room;
        for (int o = 1; o < 32; o <<= 1) {
            const int below = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += below;
        }
        s_row[lane] = rs;
        s_len[lane] = len;
        s_at[lane] = end - room;
        if (lane == 31) s_at[32] = end;
        if (lane == 0 && F.share) note_shares(slice, F.n_slices, F.off, F.share, F.blocks);
    }
    const int64_t at = F.off[slice], steps = F.off[slice + 1] - at;
    __syncthreads();
    const bool staged = s_at[32] <= F.cap;
    if (staged) {
        for (int r = warp; r < per; r += FILL_THREADS / 32) {
            const int64_t rs = s_row[r];
            const int len = s_len[r], to = s_at[r];
            for (int e = lane; e < len; e += 32) {
                if constexpr (NV > 0) {
                    VT v[NV];
                    fn(rs + e, v);
#pragma unroll
                    for (int t = 0; t < NV; t++) sv[t * F.cap + to + e] = v[t];
                }
                if (F.scol) sc[to + e] = F.col[rs + e];
            }
        }
        __syncthreads();
    }
    const int r = lane >> F.lg_l, h = lane & ((1 << F.lg_l) - 1);
    const int len = s_len[r], from = s_at[r];
    for (int64_t k = warp; k < steps; k += FILL_THREADS / 32) {
        const int64_t e = (k << F.lg_l) + h;
        const bool live = e < len;
        if constexpr (NV > 0) {
            VT v[NV];
            if (!staged && live) fn(s_row[r] + e, v);
#pragma unroll
            for (int t = 0; t < NV; t++)
                out[(at + k) * (32 * NV) + 32 * t + lane] = !live ? (VT)0 : staged ? sv[t * F.cap + from + e] : v[t];
        }
        if (F.scol) F.scol[(at + k) * 32 + lane] = !live ? -1 : staged ? sc[from + e] : F.col[s_row[r] + e];
    }
}

// Fills `out` of layout L (of the stencils themselves, no ghost rows), and its columns where they are still to come.
template <class VT, int NV, class Fn>
cudaError_t launch_sell_fill(labfm_ctx *ctx, Sell &L, VT *out, Fn fn)
{
    const bool cols = !L.valid;
    const size_t per_entry = NV * sizeof(VT) + (cols ? sizeof(int32_t) : 0);
    const int64_t want = (int64_t)(32 >> L.lg_l) * (ctx->longest | 1) + 32;
    const int cap = (int)(want * (int64_t)per_entry <= FILL_SMEM ? want : FILL_SMEM / per_entry) / 2 * 2;
    const SellFill F{ctx->n, L.n_slices, L.lg_l, cap, L.off.as<int64_t>(), ctx->row_ptr.as<int64_t>(), ctx->col.as<int32_t>(),
                     cols ? L.col.as<int32_t>() : nullptr, cols && !L.even ? L.share.as<int64_t>() : nullptr, L.blocks};
    cudaError_t e = cudaSuccess;
    if (cap * per_entry > 47 * 1024)
        e = cudaFuncSetAttribute(k_sell_fill<VT, NV, Fn>, cudaFuncAttributeMaxDynamicSharedMemorySize, FILL_SMEM);
    if (e != cudaSuccess) return e;
    k_sell_fill<VT, NV><<<(unsigned)L.n_slices, FILL_THREADS, cap * per_entry, ctx->stream>>>(F, out, fn);
    e = cudaGetLastError();
    if (e == cudaSuccess) L.valid = true;
    return e;
}

}  // namespace labfm
