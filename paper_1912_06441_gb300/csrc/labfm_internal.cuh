// Internal declarations shared by the translation units of liblabfm.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <unordered_map>

#include "labfm.h"

namespace labfm {

constexpr int KMAX = LABFM_MAX_ORDER;
constexpr int PMAX = LABFM_PMAX;
constexpr int MAX_OPS = LABFM_MAX_OPS;
// Lowest order a mixed-precision build runs through the mixed kernels; lower orders go to the
// FP64 kernel (small, well conditioned systems, exact to the FP64 floor there; above, the refined weights of the mixed
// builds are one to three orders of magnitude closer to the exact ones).
constexpr int MIXED_MIN_ORDER = 5;

__host__ __device__ constexpr int p_of_k(int k) { return (k * k + 3 * k) / 2; }

// Grow-only device buffer owned by a context.
struct DevBuf {
    void *ptr = nullptr;
    size_t bytes = 0;
    cudaError_t reserve(size_t need);
    void release();
    template <class T> T *as() const { return static_cast<T *>(ptr); }
};

// The sliced layout of the stencils (see sell.cu), built once per stencil search by the first call that reads it.
struct Sell {
    bool shaped = false;   // lg_l .. off are those of the stencils
    bool valid = false;    // ... and col and share
    int lg_l = 0;          // lanes per node, log2
    int64_t n_slices = 0;
    int64_t places = 0;    // entries with the empty places, at most
    int blocks = 0;        // shares of the slices, one per block of a run
    bool even = false;     // shares of equal numbers of slices
    bool whole = false;    // ... none of which can be worth a cut
    DevBuf off, col, steps, share;
    void release()
    {
        shaped = valid = false;
        off.release();
        col.release();
        steps.release();
        share.release();
    }
};

// Cached CUDA graph of an RK4 run, with everything its launches were recorded with: it is
// replayed only while all of these are unchanged.
struct StepGraph {
    cudaGraphExec_t exec = nullptr;
    const void *u = nullptr;
    const void *v = nullptr;  // second field (Burgers' equation)
    const void *frozen = nullptr;
    int dtype = -1;
    double dt = 0;
    int64_t nsteps = 0;
    int64_t n = -1, nnz = -1;
    int wdtype = -1;
    const void *row_ptr = nullptr, *col = nullptr, *wc = nullptr, *acc = nullptr, *sa = nullptr, *sb = nullptr;
    void release();
};

}  // namespace labfm

// Bytes of the context's host words: a wait of a run (a solve) gave up
constexpr int LABFM_GAVE_UP = 1000, LABFM_SOLVE_GAVE_UP = 1004;

struct labfm_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    int num_sms = 0;
    std::string err;

    // stencils
    int64_t n = 0;
    int64_t nnz = 0;
    int64_t longest = 0;  // entries of the longest row
    int periodic = 0;
    double lo[2] = {0, 0}, hi[2] = {0, 0};
    labfm::DevBuf node_xy, node_h;  // context copies of the node positions and h
    labfm::DevBuf row_ptr, col;
    labfm::Sell sell;  // of these stencils, for the FP64 products
    labfm::DevBuf sync_buf;  // barrier words of the cooperative runs
    int run_blocks = 0;      // blocks that fit the context's stream at once
    // scratch of the neighbour search
    labfm::DevBuf cell_of, cell_count, cell_start, cell_nodes, counts, scan_tmp, misc;

    // weights
    bool have_weights = false;
    int n_ops = 0;
    int wdtype = LABFM_F64;
    labfm::DevBuf w;
    labfm::DevBuf status_tmp;
    labfm::DevBuf wtilde;  // scratch of the mixed-precision build: unscaled weights in double
    labfm::DevBuf mscratch;  // scratch of the mixed-precision build: per-node matrices of one batch
    labfm::DevBuf mrecs;     // scratch of the mixed-precision build: per-entry preamble records
    labfm::DevBuf mwstore;   // scratch of the mixed-precision build: W of every entry (double-float)
    labfm::DevBuf mfallback; // scratch of the mixed-precision build: nodes rebuilt in FP64
    // statistics of the last labfm_build_weights (labfm_get_build_info)
    int64_t info_ref_hist[8] = {0};
    int64_t info_fp64_rebuilt = 0;
    int info_group[LABFM_MAX_ORDER + 1] = {0};  // threads per node of the FP64 kernel, per order built by it
    int info_inv_tpr[LABFM_MAX_ORDER + 1] = {0};  // threads per row of the mixed inversion, per order

    // RK4
    labfm::DevBuf wcomb, rk_acc, rk_stage_a, rk_stage_b;
    double beta_cached[LABFM_MAX_OPS] = {0};
    int wcomb_dtype = -1;
    bool wcomb_valid = false;
    labfm::StepGraph graph;
    cudaStream_t capture_stream = nullptr;  // private stream used only to record the RK4 graphs

    // RK4 of Burgers' equation: per entry (w^0, w^1, sum_{d>=2} beta_d w^d) in the weight type
    bool grad01 = false;  // operators 0 and 1 of the built weights are d/dx and d/dy
    labfm::DevBuf wburg, bu_acc, bu_stage_a, bu_stage_b;
    double beta_burg[LABFM_MAX_OPS] = {0};
    bool wburg_valid = false, wburg_sliced = false;
    labfm::StepGraph graph_burgers;

    // implicit solves (BiCGStab): operator weights in the sliced layout, eleven vectors, partial sums, and for Neumann
    // ghost rows their map and the layout with their parents' stencils
    labfm::DevBuf sol_w, sol_vec, sol_part, sol_gmap;
    labfm::Sell sell_ghost;

    // launch shapes chosen by the apply / RK4 autotuner:
    // key (kind, n_ops, dtypes, size class of n, mean stencil size) -> (G << 8) | UNR
    std::unordered_map<uint64_t, uint32_t> tuned;

    // pinned host words for status read-back; at bytes LABFM_GAVE_UP, LABFM_SOLVE_GAVE_UP: a barrier gave up
    void *host_small = nullptr;
};

namespace labfm {

labfm_status fail(labfm_ctx *ctx, labfm_status st, const std::string &msg);
labfm_status cuda_fail(labfm_ctx *ctx, cudaError_t e, const char *where);

// Exclusive prefix sum of in[0..n) into out[0..n]; out[n] = total.  `tmp` is scratch.  *largest (0 before) becomes the largest
// in[i] (non-negative); null: not wanted.
cudaError_t exclusive_scan_i32_to_i64(const int32_t *in, int64_t *out, int64_t n, DevBuf &tmp, cudaStream_t s,
                                      unsigned long long *largest = nullptr);
// The same scan on a caller-provided workspace of tmp_elems int64 (at least scan_workspace_elems(n)).
size_t scan_workspace_elems(int64_t n);
cudaError_t exclusive_scan_i32_to_i64_ws(const int32_t *in, int64_t *out, int64_t n, int64_t *tmp, size_t tmp_elems,
                                         cudaStream_t s, unsigned long long *largest = nullptr);

// Arguments of the mixed-precision build kernel (see build_mixed.cu).
struct MixedArgsPublic {
    int64_t n_list;
    const int32_t *list;
    const double *xy, *h;
    const int64_t *row_ptr;
    const int32_t *col;
    int periodic;
    double L[2], halfL[2];
    int rbf, n_ops, nref;
    int adaptive;                   // 1: refine each node until it converges, at most nref steps
    int32_t *fb_list;               // [n] nodes handed to the FP64 build (refinement diverged)
    unsigned long long *fb_count;   // device counter of fb_list
    unsigned long long *ref_hist;   // device [nref + 1]: nodes by refinement steps taken
    void *w;
    int wdtype;
    double *wt;
    int32_t *node_status;
    unsigned long long *n_bad;
    int lmax[MAX_OPS];
    double C[MAX_OPS * PMAX];
    int num_sms;
    int64_t batch_nodes;  // nodes per batch; `scratch` holds batch_nodes * mixed_scratch_bytes_per_node(k)
    void *scratch;
    void *recs;  // [nnz] per-entry records, mixed_record_bytes() each
    int tc;      // 1: moment matrices on the tensor cores (exact BF16 slices), 0: double-float
    int inv_tpr; // threads per matrix row in the inversion: 1 (rows in registers), 2 or 4
    unsigned long long *tc_timeout;  // device counter of tensor-core waits that gave up
    void *wstore;  // [nnz][p(k)] double-float W kept between the assembly and the weights, or null
};
// The mixed build of the listed nodes, all at order k (MIXED_MIN_ORDER <= k <= KMAX).
cudaError_t launch_build_mixed(int k, const MixedArgsPublic &p, cudaStream_t s);
size_t mixed_scratch_bytes_per_node(int k);
size_t mixed_record_bytes();

// The sliced layout as kernels read it
struct SellView {
    int64_t n_slices;
    const int64_t *off;
    const int32_t *col;
    const int64_t *share;  // [blocks + 1]: the slices of share b are share[b] .. share[b + 1] - 1; null: equal numbers,
    int each, more;        // `each`, and `more` in all besides, spread evenly
    unsigned recip;        // 2^32 / blocks, rounded up
    int blocks;
    int lg_l;
    bool whole;            // no block can have a slice to cut
};

// The scale on which sweeps are shared out: slice s takes [slice_at(s), slice_at(s + 1)), a place for each of its steps and
// SLICE_COST for the update of its nodes (a step is two FP64 instructions or more, an update four and two per combining step).
constexpr int SLICE_COST = 4;
#ifdef __CUDACC__
// A lane's place in the sliced layout: node i (-1: none) and entry k L + h of its row at step k
struct SellLane {
    int64_t i = -1, at = 0;
    int steps = 0, h;
    SellLane() = default;
    __device__ SellLane(int64_t slice, int lane, int64_t n, const SellView &S)
    {
        h = lane & ((1 << S.lg_l) - 1);
        if (slice >= S.n_slices) return;
        const int64_t node = slice * (32 >> S.lg_l) + (lane >> S.lg_l);
        if (node < n) i = node;
        at = S.off[slice] * 32 + lane;
        steps = (int)(S.off[slice + 1] - S.off[slice]);
    }
    // so many steps from place `from` on
    __device__ SellLane(int64_t slice, int64_t from, int count, int lane, int64_t n, const SellView &S) : at(from * 32 + lane), steps(count)
    {
        h = lane & ((1 << S.lg_l) - 1);
        const int64_t node = slice * (32 >> S.lg_l) + (lane >> S.lg_l);
        if (node < n) i = node;
    }
};

// A slice's steps U at a time: indices and weights (NW of them per entry, 32 places apart) in registers, loaded ahead.
template <int U, int NW, class VT>
struct SliceBatch {
    int c[U];
    VT w[U][NW];
    // steps k0 .. k0 + U - 1 of lane l's slice; c = -1 where there is no entry
    __device__ __forceinline__ void load(const SellLane &l, int lane, int k0, const SellView &S, const VT *__restrict__ wc)
    {
        const int64_t at = l.at + 32 * (int64_t)k0;
        const VT *wr = wc + NW * (at - lane) + lane;
#pragma unroll
        for (int q = 0; q < U; q++) {
            c[q] = -1;
            if (k0 + q < l.steps) {
                c[q] = __ldcs(S.col + at + 32 * q);
#pragma unroll
                for (int t = 0; t < NW; t++) w[q][t] = __ldcs(wr + 32 * (NW * q + t));
            }
        }
    }
};

// A slice's sums by one lane: indices and weights are loaded two batches of U steps ahead and the values they name
// (NX of them per entry) gathered one batch ahead.  The warps of a block go in step through the FP64 pipe, so that
// without that they all wait for each batch's gathers at the same time (0.35 us a batch).
template <int U, int NW, int NX, class VT>
struct SlicePipe {
    SliceBatch<U, NW, VT> cur, nxt;
    __device__ __forceinline__ void preload(const SellLane &l, int lane, const SellView &S, const VT *__restrict__ wc)
    {
        cur.load(l, lane, 0, S, wc);
        nxt.load(l, lane, U, S, wc);
    }
    // gather(j, x) and add(q, x, w) for every entry of the lane; preload comes first
    template <class Gather, class Add>
    __device__ __forceinline__ void run(const SellLane &l, int lane, const SellView &S, const VT *__restrict__ wc, Gather gather,
                                        Add add)
    {
        double x[U][NX], xn[U][NX];
#pragma unroll
        for (int q = 0; q < U; q++)
            if (cur.c[q] >= 0) gather(cur.c[q], x[q]);
        for (int k0 = 0; k0 < l.steps; k0 += U) {
#pragma unroll
            for (int q = 0; q < U; q++)
                if (nxt.c[q] >= 0) gather(nxt.c[q], xn[q]);
            SliceBatch<U, NW, VT> far;
            far.load(l, lane, k0 + 2 * U, S, wc);
#pragma unroll
            for (int q = 0; q < U; q++)
                if (cur.c[q] >= 0) add(q, x[q], cur.w[q]);
            cur = nxt;
            nxt = far;
#pragma unroll
            for (int q = 0; q < U; q++)
#pragma unroll
                for (int t = 0; t < NX; t++) x[q][t] = xn[q][t];
        }
    }
};

// Runs of many dependent sweeps over a node set (RK4 steps, solver iterations) as one cooperative launch: a block per
// SM, a barrier over the grid between sweeps.  Launched one by one a sweep of a small set costs its launch and its
// uneven last blocks again as much as its sums.  What a sweep writes for others to read carries no __restrict__ in the
// kernel: it is not constant data of the launch.
constexpr int RUN_THREADS = 512;
constexpr int RUN_WARPS = RUN_THREADS / 32;
struct GridSync {
    unsigned *count;    // device: arrivals, 0 at the launch; then 1 once a wait gave up, until the host has reported it
    unsigned *gave_up;  // pinned host word, set where a wait gave up
};
// Reads of the count that a wait makes before it gives up: of the order of a second.  Set at compile time for tests (a
// limit that came with the launch cost 0.05 to 0.1 us a barrier).
#ifndef LABFM_SYNC_POLLS
#define LABFM_SYNC_POLLS (1u << 21)
#endif
constexpr unsigned SYNC_POLLS = LABFM_SYNC_POLLS;

struct GridBarrier {
    GridSync g;
    unsigned target = 0;
    // Whether an earlier run, or a block of this one, gave up: the fields are not valid, and the run leaves them as they
    // are.  check comes before a block barrier, stopped behind it.
    static __device__ __forceinline__ int &stop_word()
    {
        __shared__ int s_stop;
        return s_stop;
    }
    __device__ __forceinline__ void check() const
    {
        if (threadIdx.x == 0) stop_word() = *(volatile unsigned *)(g.count + 1) != 0;
    }
    static __device__ __forceinline__ bool stopped() { return stop_word() != 0; }
    // Waits until every block has arrived; what they wrote before is visible after.  false: a block did not arrive
    // within SYNC_POLLS reads (or another block has found so): the caller returns.
    __device__ bool wait()
    {
        __shared__ int s_ok;
        __syncthreads();
        if (threadIdx.x == 0) {
            target += gridDim.x;
            // (releases the whole block's writes: the barrier above orders them before it)
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(g.count) : "memory");
            int ok = 1;
            unsigned now, polls = 0;
            while (true) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(g.count) : "memory");
                if ((int)(now - target) >= 0) break;
                if (++polls >= SYNC_POLLS || ((polls & 255u) == 0 && *(volatile unsigned *)(g.count + 1))) {
                    *(volatile unsigned *)(g.count + 1) = 1u;
                    *(volatile unsigned *)g.gave_up = 1u;
                    __threadfence_system();
                    ok = 0;
                    break;
                }
            }
            s_ok = ok;
        }
        __syncthreads();
        return s_ok != 0;
    }
};

__device__ __forceinline__ int64_t slice_at(const SellView &S, int64_t s) { return S.off[s] + SLICE_COST * s; }

// This block's slices [first, last): its share, or where the grid has fewer blocks than shares, several
__device__ __forceinline__ void block_share(const SellView &S, int64_t &first, int64_t &last)
{
    int b0 = blockIdx.x, b1 = blockIdx.x + 1;
    if (gridDim.x != S.blocks) {
        b0 = b0 * S.blocks / gridDim.x;
        b1 = b1 * S.blocks / gridDim.x;
    }
    if (S.share) {
        first = S.share[b0];
        last = S.share[b1];
    } else {
        // (b more / blocks, by the reciprocal: exact up to some 250 blocks)
        first = (int64_t)S.each * b0 + __umulhi((unsigned)(S.more * b0), S.recip);
        last = (int64_t)S.each * b1 + __umulhi((unsigned)(S.more * b1), S.recip);
    }
}

// A warp's part of its block's slices: every RUN_WARPS-th slice, or where that gives some warp CUT_COST places more than an
// equal part (every barrier waits for the last warp), one of RUN_WARPS equal runs of the block's places, cut within
// slices too.  Then the warp in whose run a slice begins updates its nodes, and the warps that the slice runs on into
// add up their part of it.  Order 4, 289^2 nodes, 18 slices of 49 steps a block: 27.4 us a stage in two rounds of whole slices, 21.1
// cut (24.4 as launches); 257^2, 14 slices: 16.3 and 16.8; 161^2, 11 slices of 25 steps: 7.9 and 8.8; 41^2, 3 of 7: 3.2 and 3.5.
// CUT_COST is what those and 25 more sizes between 41^2 and 900^2 come to: a second piece's loads and a block barrier.
constexpr int CUT_COST = 25;
struct WarpShare {
    int64_t from;             // its first piece: the place where it begins
    int steps;                // ... and its steps
    int first, last, stride;  // the slices this warp updates: first, first + stride, ... below last
    bool head;                // the first piece is a part of slice first - 1, which another warp updates
    bool cut;                 // some slice of the block is shared by warps
    int open;                 // it adds up the first `open` steps of slice last - 1 itself; < 0: all of them
    int parts;                // ... and so many warps after it add up the rest
};
// This warp's part, kept in shared memory: read once a piece, where registers are short
__device__ __forceinline__ WarpShare &warp_share()
{
    __shared__ WarpShare s_share[RUN_WARPS];
    return s_share[threadIdx.x >> 5];
}
// Forms the parts of the block's warps; all of its threads take part.
__device__ __forceinline__ void share_out(const SellView &S, int64_t s0, int64_t s1)
{
    __shared__ int s_first[RUN_WARPS + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto whole_slices = [&] {
        const int64_t t = s0 + warp;
        if (lane == 0)
            warp_share() = t < s1 ? WarpShare{S.off[t], (int)(S.off[t + 1] - S.off[t]), (int)t, (int)s1, RUN_WARPS, false, false, -1, 0}
                                  : WarpShare{0, 0, (int)t, (int)t, RUN_WARPS, false, false, -1, 0};
    };
    if (S.whole) {  // (a run of two steps on 64^2 nodes would take 7 % longer for finding that out)
        whole_slices();
        __syncthreads();
        return;
    }
    const int64_t base = slice_at(S, s0), total = slice_at(S, s1) - base;
    int64_t whole = 0;  // places of every RUN_WARPS-th slice
    for (int64_t t = s0 + warp + RUN_WARPS * lane; t < s1; t += RUN_WARPS * 32) whole += slice_at(S, t + 1) - slice_at(S, t);
    for (int o = 16; o > 0; o >>= 1) whole += __shfl_xor_sync(0xffffffffu, whole, o);
    if (!__syncthreads_or(whole > total / RUN_WARPS + CUT_COST)) {
        whole_slices();
        __syncwarp();
        return;
    }
    const int64_t a = base + total * warp / RUN_WARPS, z = base + total * (warp + 1) / RUN_WARPS;
    // the first slice at or behind a, a 32nd of what is left at a time
    int64_t lo = s0, hi = s1;
    while (lo < hi) {
        const int64_t gap = (hi - lo + 31) / 32, at = lo + gap * lane;
        const int before = __popc(__ballot_sync(0xffffffffu, at < hi && slice_at(S, at) < a));
        hi = min(hi, lo + gap * before);
        if (before > 0) lo += gap * (before - 1) + 1;
    }
    if (lane == 0) s_first[warp] = (int)lo;
    if (threadIdx.x == 0) s_first[RUN_WARPS] = (int)s1;
    __syncthreads();
    WarpShare W{0, 0, (int)lo, s_first[warp + 1], 1, false, false, -1, 0};
    if (W.last > W.first) {
        const int64_t at = slice_at(S, W.last - 1), steps = S.off[W.last] - S.off[W.last - 1];
        if (z - at < steps) {
            W.open = (int)(z - at);
            while (warp + 1 + W.parts < RUN_WARPS && base + total * (warp + 1 + W.parts) / RUN_WARPS - at < steps) W.parts++;
        }
        W.from = S.off[W.first];
        W.steps = W.open >= 0 && W.last - W.first == 1 ? W.open : (int)(S.off[W.first + 1] - W.from);
    }
    if (W.first > s0) {
        const int64_t at = slice_at(S, W.first - 1), steps = S.off[W.first] - S.off[W.first - 1];
        if (a - at < steps) {
            W.head = true;
            W.from = S.off[W.first - 1] + (a - at);
            W.steps = (int)(min(steps, z - at) - (a - at));
        }
    }
    W.cut = __syncthreads_or(W.open >= 0) != 0;
    if (lane == 0) warp_share() = W;
    __syncwarp();
}

// Where the warps leave their parts of others' slices
template <int NS>
__device__ __forceinline__ double (&left_parts())[RUN_WARPS][NS][32]
{
    __shared__ double s_part[RUN_WARPS][NS][32];
    return s_part;
}

// A block's sweep over its slices, NS sums per lane.  With a slice's node values by begin(lane, whether this warp updates it):
// gather and add as in SlicePipe (add with those values), part(values, sums) the lane's sums, and where the warp
// updates the slice finish(lane, values, sums) with the parts of all warps.  Every thread of the block takes part, after
// share_out; a block barrier has to follow before the next run.
// KEEP: the first piece is kept in registers, found by place() once or, where registers are short, before every preload; else it
// is read again from the warp's share.  (Burgers runs are 3 to 4 % faster without, 161^2: 68.4 us a step against 70.4; heat
// and solves up to 4 % with, 41^2: 11.9 us a step against 12.5.)
template <int U, int NW, int NX, int NS, bool KEEP, class VT>
struct SliceSweep {
    SlicePipe<U, NW, NX, VT> pipe;
    SellLane kept_at;
    int kept_slice;
    bool kept_mine, kept_last;  // this warp updates it; it has no further one

    // the first piece (of none: no node and no step)
    static __device__ __forceinline__ SellLane begin_at(int64_t n, const SellView &S)
    {
        const WarpShare &W = warp_share();
        const bool any = W.head || W.first < W.last;
        return SellLane(any ? W.first - W.head : S.n_slices, W.from, W.steps, threadIdx.x & 31, n, S);
    }
    __device__ __forceinline__ void place(int64_t n, const SellView &S)
    {
        static_assert(KEEP, "nothing is kept");
        const WarpShare &W = warp_share();
        kept_slice = W.first - W.head;
        kept_mine = kept_slice >= W.first && kept_slice < W.last;
        kept_last = kept_slice + W.stride >= W.last;
        kept_at = begin_at(n, S);
    }
    // the first loads of the next run
    __device__ __forceinline__ void preload(int64_t n, const SellView &S, const VT *__restrict__ wc)
    {
        if constexpr (KEEP) pipe.preload(kept_at, threadIdx.x & 31, S, wc);
        else pipe.preload(begin_at(n, S), threadIdx.x & 31, S, wc);
    }
    template <class Begin, class Gather, class Add, class Part, class Finish>
    __device__ __forceinline__ void run(int64_t n, const SellView &S, const VT *__restrict__ wc, Begin begin, Gather gather,
                                        Add add, Part part, Finish finish)
    {
        double(&s_part)[RUN_WARPS][NS][32] = left_parts<NS>();
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const WarpShare &W = warp_share();
        SellLane l;
        int slice;
        bool mine, last;
        if constexpr (KEEP) {
            l = kept_at;
            slice = kept_slice;
            mine = kept_mine;
            last = kept_last;
        } else {
            l = begin_at(n, S);
            slice = W.first - W.head;
        }
        while (true) {  // a warp without a piece goes through once, for the barrier
            if constexpr (!KEEP) {
                mine = slice >= W.first && slice < W.last;
                last = slice + W.stride >= W.last;
            }
            auto v = begin(l, mine);
            double p[NS];
            pipe.run(l, lane, S, wc, gather, [&](int q, const double(&x)[NX], const VT(&w)[NW]) { add(v, q, x, w); });
            part(v, p);
            if (W.cut) {
                if (!mine)
#pragma unroll
                    for (int t = 0; t < NS; t++) s_part[warp][t][lane] = p[t];
                if (last) __syncthreads();  // every warp once
                if (mine && last && W.open >= 0)
                    for (int k = 1; k <= W.parts; k++)
#pragma unroll
                        for (int t = 0; t < NS; t++) p[t] += s_part[warp + k][t][lane];
            }
            if (mine) finish(l, v, p);
            if (last) break;
            slice += W.stride;
            if constexpr (KEEP) {
                mine = true;
                last = slice + W.stride >= W.last;
            }
            l = SellLane(slice, lane, n, S);
            if (slice + 1 == W.last && W.open >= 0) l.steps = W.open;
            pipe.preload(l, lane, S, wc);
        }
    }
};

// Cooperative launch of such a run on the context's stream.  Its blocks have to fit the SMs together: where the stream has
// fewer of them than the device (a green context, a share of the device), with half as many blocks, and so on.
template <class... P, class... A>
cudaError_t launch_run(labfm_ctx *ctx, const SellView &S, void (*kern)(P...), A... args)
{
    cudaError_t e = cudaMemsetAsync(ctx->sync_buf.ptr, 0, sizeof(unsigned), ctx->stream);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(RUN_THREADS);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    while (true) {
        cfg.gridDim = dim3((unsigned)(S.blocks < ctx->run_blocks ? S.blocks : ctx->run_blocks));
        e = cudaLaunchKernelEx(&cfg, kern, P(args)...);
        if (e != cudaErrorCooperativeLaunchTooLarge || cfg.gridDim.x == 1) return e;
        cudaGetLastError();
        ctx->run_blocks = (int)(cfg.gridDim.x + 1) / 2;
    }
}
// The barrier words, before the first launch
inline cudaError_t ensure_sync(labfm_ctx *ctx)
{
    if (ctx->sync_buf.ptr) return cudaSuccess;
    const cudaError_t e = ctx->sync_buf.reserve(256);
    return e == cudaSuccess ? cudaMemsetAsync(ctx->sync_buf.ptr, 0, 256, ctx->stream) : e;
}
inline unsigned *gave_up_word(const labfm_ctx *ctx, int byte)
{
    return reinterpret_cast<unsigned *>(static_cast<char *>(ctx->host_small) + byte);
}
inline GridSync grid_sync(const labfm_ctx *ctx, int byte)
{
    return GridSync{ctx->sync_buf.as<unsigned>(), gave_up_word(ctx, byte)};
}
#endif
// Whether a wait of a run (byte LABFM_GAVE_UP) or solve that has ended gave up; launches from here on run again.
inline bool gave_up(labfm_ctx *ctx, int byte)
{
    volatile unsigned *w = reinterpret_cast<unsigned *>(static_cast<char *>(ctx->host_small) + byte);
    if (*w == 0) return false;
    *w = 0;
    cudaMemsetAsync(ctx->sync_buf.as<unsigned>() + 1, 0, sizeof(unsigned), ctx->stream);
    return true;
}
inline labfm_status run_gave_up(labfm_ctx *ctx)
{
    return gave_up(ctx, LABFM_GAVE_UP)
               ? fail(ctx, LABFM_ERR_TIMEOUT, "a wait between the blocks of an earlier run gave up: the fields of the runs since are not valid")
               : LABFM_OK;
}
inline SellView sell_view(const Sell &L)
{
    const int each = (int)(L.n_slices / L.blocks), more = (int)(L.n_slices % L.blocks);
    const unsigned recip = (unsigned)(((1ull << 32) + L.blocks - 1) / L.blocks);  // (one block: 0, and more = 0)
    return SellView{L.n_slices, L.off.as<int64_t>(), L.col.as<int32_t>(), L.even ? nullptr : L.share.as<int64_t>(), each, more,
                    recip, L.blocks, L.lg_l, L.whole};
}
labfm_status ensure_sell_shape(labfm_ctx *ctx);  // ctx->sell of the current stencils, col and share still to come (sell_fill.cuh)
labfm_status ensure_sell(labfm_ctx *ctx);        // all of it
// The layout of the stencils with the rows in gmap (>= 0: a Neumann ghost row) replaced by their parents' (gmap null: none)
labfm_status build_sell(labfm_ctx *ctx, Sell &L, const int32_t *gmap, const int64_t *parent);

// Kernel launchers (each returns the launch error).
labfm_status run_neighbours(labfm_ctx *ctx, int64_t n, const double *xy, const double *h, int periodic,
                            const double lo[2], const double hi[2], int64_t *nnz_out);
labfm_status run_build(labfm_ctx *ctx, const int8_t *order, int uniform_order, int rbf, int n_ops, const double *C,
                       int precision, int weight_dtype, int32_t *node_status, int64_t *n_bad_out);
cudaError_t launch_apply(labfm_ctx *ctx, uint32_t op_mask, const void *f, int field_dtype, void *out);
// Neumann ghost rows of an implicit solve (Sec. 5.2); n_ghost = 0: none
struct SolveNeumann {
    int64_t n_ghost = 0;
    const int64_t *ghost = nullptr, *parent = nullptr;  // device [n_ghost]
    const double *normal = nullptr;                     // device [n_ghost][2]
    int op_x = 0, op_y = 0;
};
labfm_status run_solve(labfm_ctx *ctx, int op, const double *f, double *phi, const uint8_t *dirichlet,
                       const SolveNeumann &nm, double tol, int max_iter, int *iters_out, double *resid_out);
labfm_status run_step_burgers(labfm_ctx *ctx, const double *beta, void *u, void *v, int field_dtype, double dt,
                              int64_t nsteps, const uint8_t *frozen);
labfm_status run_step(labfm_ctx *ctx, const double *beta, void *u, int field_dtype, double dt, int64_t nsteps,
                      const uint8_t *frozen);

}  // namespace labfm

#define LABFM_CUDA_TRY(ctx, expr)                                   \
    do {                                                            \
        cudaError_t e_ = (expr);                                    \
        if (e_ != cudaSuccess) return labfm::cuda_fail(ctx, e_, #expr); \
    } while (0)
