// FP64 weight build (Sec. 3.1-3.2), the host side: the choice of the group size per order, the bucketing of
// per-node orders, and the routing of a mixed build's orders (device side: build_node.cuh).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "build_node.cuh"

namespace labfm {
namespace {

// Bucketing by (order, stencil size), both descending: key = (KMAX - k) 256 + 255 - min(N_i, 255).
constexpr int NBUCKET = (KMAX + 1) * 256;
__device__ __forceinline__ int bucket_key(int k, int64_t deg) { return (KMAX - k) * 256 + 255 - (int)min(deg, (int64_t)255); }

__global__ void k_bucket_count(int64_t n, const int8_t *__restrict__ order, const int64_t *__restrict__ row_ptr,
                               unsigned int *__restrict__ hist, unsigned long long *__restrict__ bad)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = order[i];
    if (k < 1 || k > KMAX) {
        atomicAdd(bad, 1ull);
        return;
    }
    atomicAdd(&hist[bucket_key(k, row_ptr[i + 1] - row_ptr[i])], 1u);
}

// cursor[b] starts at the first list position of bucket b
__global__ void k_bucket_scatter(int64_t n, const int8_t *__restrict__ order, const int64_t *__restrict__ row_ptr,
                                 unsigned int *__restrict__ cursor, int32_t *__restrict__ list)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = order[i];
    if (k < 1 || k > KMAX) return;
    list[atomicAdd(&cursor[bucket_key(k, row_ptr[i + 1] - row_ptr[i])], 1u)] = (int32_t)i;
}

// the full chain rule of D(W0) in the elements of degrees 2 and 3
bool chain_rule(int rbf) { return (rbf & LABFM_ABF_DW0_ONLY) == 0; }

cudaError_t launch_fp64_order(int k, int G, const BuildArgs &a, int num_sms, cudaStream_t s)
{
    return (k >= FORM_MIN_ORDER && chain_rule(a.rbf) ? launch_order_chain : launch_order_dw0)(k, G, a, num_sms, s);
}

}  // namespace

// Refinement steps of a mixed build: LABFM_PREC_MIXED[_TC]_REFINE(n) fixes n; otherwise each
// node refines until it converges (at most NREF_ADAPTIVE steps; one for most nodes).
constexpr int NREF_ADAPTIVE = 6;
static int precision_nref(int precision, bool &adaptive)
{
    int forced = (precision >> 8) & 0xf;  // LABFM_PREC_MIXED_REFINE(n) stores n + 1 here
    adaptive = forced == 0;
    return forced ? forced - 1 : NREF_ADAPTIVE;
}

// LABFM_MIXED_INVERSION = registers | shared2 | shared4 fixes the form of the mixed builds'
// inversion (rows in registers; 2 or 4 threads per row in shared memory) instead of the build
// autotuner's choice (diagnostics and tests); unset or any other value: the autotuner decides.
static int mixed_inversion_override()
{
    const char *v = std::getenv("LABFM_MIXED_INVERSION");
    if (!v) return 0;
    if (std::strcmp(v, "registers") == 0) return 1;
    if (std::strcmp(v, "shared2") == 0) return 2;
    if (std::strcmp(v, "shared4") == 0) return 4;
    return 0;
}

labfm_status run_build(labfm_ctx *ctx, const int8_t *order, int uniform_order, int rbf, int n_ops, const double *Cin,
                       int precision, int weight_dtype, int32_t *node_status, int64_t *n_bad_out)
{
    cudaStream_t s = ctx->stream;
    const int64_t n = ctx->n;
    const int base_prec = precision & 0xff;
    const bool mixed = base_prec == LABFM_PREC_MIXED || base_prec == LABFM_PREC_MIXED_TC;
    const bool chain = chain_rule(rbf);
    size_t wbytes = (size_t)ctx->nnz * n_ops * (weight_dtype == LABFM_F64 ? 8 : 4);
    LABFM_CUDA_TRY(ctx, ctx->w.reserve(wbytes > 0 ? wbytes : 8));
    if (mixed) LABFM_CUDA_TRY(ctx, ctx->wtilde.reserve((size_t)ctx->nnz * n_ops * 8 + 8));
    // misc layout: [0] bad nodes, [1] bad orders, [30] tensor-core waits that gave up, [31] nodes
    // handed to the FP64 build, [32..39] nodes by refinement steps; from byte 1024 the bucket
    // histogram, from byte 1024 + 4 NBUCKET the bucket cursors
    constexpr int NMISC = 40;
    LABFM_CUDA_TRY(ctx, ctx->misc.reserve(1024 + 8 * (size_t)NBUCKET));
    unsigned long long *dmisc = ctx->misc.as<unsigned long long>();
    unsigned int *d_hist = reinterpret_cast<unsigned int *>(ctx->misc.as<char>() + 1024);
    unsigned int *d_cursor = d_hist + NBUCKET;
    LABFM_CUDA_TRY(ctx, cudaMemsetAsync(dmisc, 0, NMISC * sizeof(unsigned long long), s));
    for (int t = 0; t < 8; t++) ctx->info_ref_hist[t] = 0;
    for (int t = 0; t <= KMAX; t++) ctx->info_group[t] = ctx->info_inv_tpr[t] = 0;
    ctx->info_fp64_rebuilt = 0;

    BuildArgs a{};
    a.xy = ctx->node_xy.as<double>();
    a.h = ctx->node_h.as<double>();
    a.row_ptr = ctx->row_ptr.as<int64_t>();
    a.col = ctx->col.as<int32_t>();
    a.periodic = ctx->periodic;
    for (int d = 0; d < 2; d++) {
        a.L[d] = ctx->hi[d] - ctx->lo[d];
        a.halfL[d] = 0.5 * a.L[d];
    }
    a.rbf = rbf;
    a.n_ops = n_ops;
    a.w = ctx->w.ptr;
    a.wdtype = weight_dtype;
    a.node_status = node_status;
    a.n_bad = dmisc;
    for (int t = 0; t < n_ops * PMAX; t++) a.C[t] = Cin[t];

    MixedArgsPublic m{};
    if (mixed) {
        m.xy = a.xy;
        m.h = a.h;
        m.row_ptr = a.row_ptr;
        m.col = a.col;
        m.periodic = a.periodic;
        for (int d = 0; d < 2; d++) {
            m.L[d] = a.L[d];
            m.halfL[d] = a.halfL[d];
        }
        m.rbf = rbf;
        m.n_ops = n_ops;
        m.w = a.w;
        m.wdtype = weight_dtype;
        m.wt = ctx->wtilde.as<double>();
        m.node_status = node_status;
        m.n_bad = dmisc;
        m.num_sms = ctx->num_sms;
        m.tc = base_prec == LABFM_PREC_MIXED_TC;
        m.tc_timeout = dmisc + 30;
        m.fb_count = dmisc + 31;
        m.ref_hist = dmisc + 32;
        LABFM_CUDA_TRY(ctx, ctx->mfallback.reserve(sizeof(int32_t) * (n > 0 ? n : 1)));
        m.fb_list = ctx->mfallback.as<int32_t>();
        for (int t = 0; t < n_ops * PMAX; t++) m.C[t] = Cin[t];
        for (int d = 0; d < n_ops; d++) {
            int l = 0;
            for (int e = 0; e < PMAX; e++)
                if (Cin[d * PMAX + e] != 0.0) l = std::max(l, (int)elem_degree(e));
            m.lmax[d] = l;
        }
    }
    // Orders that the FP64 kernel builds: all of them for LABFM_PREC_FP64; for the mixed builds the
    // orders below MIXED_MIN_ORDER, whose p x p systems (p <= 14) are small and well conditioned:
    // there the cost is latency, which the grouped FP64 kernel hides better than the four-kernel
    // mixed pipeline, and FP64 arithmetic is accurate to the floor.  (From moments the FP64 kernel is the faster one at
    // the orders above too, 23.5 against 29.6 and 30.7 ms at order 6, 56.2 against 69.7 and 63.3 at order 8, 512^2 nodes;
    // there the mixed builds stay for the accuracy that their refinement asks for: errors at order 8 of 1e-12 against
    // 2e-9 in the median.)
    auto fp64_route = [&](int k) { return !mixed || k < MIXED_MIN_ORDER; };

    // Group size of the FP64 kernel per order: timed once per (order, mean stencil size, n_ops)
    // on up to 16,384 of the order's real nodes (the autotuner of the build), kept in the
    // context's table.  Not while the caller's stream is being captured, nor below 4,096 nodes.
    // (The form of the ABFs is not in the key, and the untimed choice of a small set is kept: both forms' timings come out
    // as that choice, 64 threads at orders 1 to 4, 128 at 5 and 6, at 200^2 nodes.)
    auto group_for = [&](int k, const int32_t *list, int64_t cnt, double deg, int &G) -> cudaError_t {
        G = k <= 4 ? 64 : (k <= 6 ? 128 : 256);
        const uint64_t dkey = (uint64_t)std::min(deg + 0.5, 65535.0);
        const uint64_t key = (dkey << 40) | ((uint64_t)k << 32) | (5ull << 24) | ((uint64_t)n_ops << 16);
        auto it = ctx->tuned.find(key);
        if (it != ctx->tuned.end()) {
            G = (int)it->second;
            return cudaSuccess;
        }
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        cudaError_t e = cudaStreamIsCapturing(s, &cap);
        if (e != cudaSuccess) return e;
        if (cap != cudaStreamCaptureStatusNone) return cudaSuccess;
        const int n_ok = (int)group_ok(k, 64) + (int)group_ok(k, 128) + (int)group_ok(k, 256);
        if (n_ok == 1) G = 256;  // one candidate: nothing to time
        if (cnt >= 4096 && n_ok > 1) {
            const int cand[3] = {64, 128, 256};
            float best = 1e30f;
            cudaEvent_t e0, e1;
            if ((e = cudaEventCreate(&e0)) != cudaSuccess) return e;
            if ((e = cudaEventCreate(&e1)) != cudaSuccess) {
                cudaEventDestroy(e0);
                return e;
            }
            BuildArgs t = a;
            t.list = list;
            t.n_list = std::min<int64_t>(cnt, 16384);
            for (int c = 0; c < 3 && e == cudaSuccess; c++) {
                if (!group_ok(k, cand[c])) continue;
                e = launch_fp64_order(k, cand[c], t, ctx->num_sms, s);  // warm-up
                if (e == cudaSuccess) e = cudaEventRecord(e0, s);
                if (e == cudaSuccess) e = launch_fp64_order(k, cand[c], t, ctx->num_sms, s);
                if (e == cudaSuccess) e = cudaEventRecord(e1, s);
                float ms = 0.0f;
                if (e == cudaSuccess) e = cudaEventSynchronize(e1);
                if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                if (e == cudaSuccess && ms < best) {
                    best = ms;
                    G = cand[c];
                }
            }
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            if (e != cudaSuccess) return e;
        }
        ctx->tuned[key] = (uint32_t)G;
        return cudaSuccess;
    };
    // the mixed kernels over the listed nodes, all at order k
    auto launch_mixed_raw = [&](int k, const int32_t *list, int64_t n_list, int tpr) -> cudaError_t {
        m.list = list;
        m.n_list = n_list;
        m.inv_tpr = tpr;
        bool adaptive = false;
        m.nref = precision_nref(precision, adaptive);
        m.adaptive = adaptive ? 1 : 0;
        // per-node matrices of one batch: at most 2^20 nodes (16 GB at k = 8)
        m.batch_nodes = std::max<int64_t>(1, std::min<int64_t>(n_list, (int64_t)1 << 20));
        cudaError_t e = ctx->mscratch.reserve(mixed_scratch_bytes_per_node(k) * (size_t)m.batch_nodes + 256);
        if (e != cudaSuccess) return e;
        m.scratch = ctx->mscratch.ptr;
        e = ctx->mrecs.reserve(mixed_record_bytes() * (size_t)ctx->nnz + 256);
        if (e != cudaSuccess) return e;
        m.recs = ctx->mrecs.ptr;
        // W of every entry, kept from the assembly for the weights kernel (8 bytes per element);
        // above 24 GB the weights kernel evaluates W again instead
        const size_t wbytes_k = (size_t)8 * p_of_k(k) * (size_t)ctx->nnz;
        m.wstore = nullptr;
        if (wbytes_k <= ((size_t)24 << 30) && ctx->mwstore.reserve(wbytes_k + 256) == cudaSuccess)
            m.wstore = ctx->mwstore.ptr;
        else
            cudaGetLastError();  // a failed reservation only disables the store
        return launch_build_mixed(k, m, s);
    };
    // Threads per row of the mixed inversion (2 or 4), timed once per (order, mean stencil size,
    // n_ops, precision) on the whole mixed pipeline over up to 16,384 of the order's nodes (the
    // timing runs' counters are cleared afterwards; their weights are overwritten by the build).
    auto launch_mixed = [&](int k, const int32_t *list, int64_t cnt, double deg) -> cudaError_t {
        // untimed (small or captured builds): rows in registers, the form that won every timing
        int tpr = 1;
        const int forced = mixed_inversion_override();
        if (forced) {
            ctx->info_inv_tpr[k] = forced;
            return launch_mixed_raw(k, list, cnt, forced);
        }
        const uint64_t dkey = (uint64_t)std::min(deg + 0.5, 65535.0);
        const uint64_t key = (dkey << 40) | ((uint64_t)k << 32) | (6ull << 24) | ((uint64_t)n_ops << 16) |
                             ((uint64_t)base_prec << 8);
        auto it = ctx->tuned.find(key);
        cudaError_t e = cudaSuccess;
        if (it != ctx->tuned.end()) {
            tpr = (int)it->second;
        } else {
            cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
            e = cudaStreamIsCapturing(s, &cap);
            if (e != cudaSuccess) return e;
            if (cap == cudaStreamCaptureStatusNone && cnt >= 4096) {
                cudaEvent_t e0, e1;
                if ((e = cudaEventCreate(&e0)) != cudaSuccess) return e;
                if ((e = cudaEventCreate(&e1)) != cudaSuccess) {
                    cudaEventDestroy(e0);
                    return e;
                }
                const int64_t nt = std::min<int64_t>(cnt, 16384);
                float best = 1e30f;
                const int cands[3] = {1, 2, 4};  // threads per row: 1 = rows in registers
                for (int ci = 0; ci < 3 && e == cudaSuccess; ci++) {
                    const int cand = cands[ci];
                    e = launch_mixed_raw(k, list, nt, cand);  // warm-up
                    if (e == cudaSuccess) e = cudaEventRecord(e0, s);
                    if (e == cudaSuccess) e = launch_mixed_raw(k, list, nt, cand);
                    if (e == cudaSuccess) e = cudaEventRecord(e1, s);
                    float ms = 0.0f;
                    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
                    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                    if (e == cudaSuccess && ms < best) {
                        best = ms;
                        tpr = cand;
                    }
                }
                cudaEventDestroy(e0);
                cudaEventDestroy(e1);
                if (e != cudaSuccess) return e;
                // the timing runs' flags, rebuild lists and step counts
                e = cudaMemsetAsync(dmisc, 0, sizeof(unsigned long long), s);
                if (e == cudaSuccess) e = cudaMemsetAsync(dmisc + 30, 0, 10 * sizeof(unsigned long long), s);
                if (e != cudaSuccess) return e;
            }
            ctx->tuned[key] = (uint32_t)tpr;
        }
        ctx->info_inv_tpr[k] = tpr;
        return launch_mixed_raw(k, list, cnt, tpr);
    };

    unsigned long long *hs = (unsigned long long *)ctx->host_small;
    if (!order) {
        const int k = uniform_order;
        if (fp64_route(k)) {
            int G = 256;
            LABFM_CUDA_TRY(ctx, group_for(k, nullptr, n, n > 0 ? (double)ctx->nnz / (double)n : 0.0, G));
            ctx->info_group[k] = G;
            LABFM_CUDA_TRY(ctx, cudaMemsetAsync(dmisc, 0, sizeof(unsigned long long), s));  // the timing runs' flags
            a.list = nullptr;
            a.n_list = n;
            LABFM_CUDA_TRY(ctx, launch_fp64_order(k, G, a, ctx->num_sms, s));
        } else {
            LABFM_CUDA_TRY(ctx, launch_mixed(k, nullptr, n, n > 0 ? (double)ctx->nnz / (double)n : 0.0));
        }
    } else {
        // bucket the nodes by (order, stencil size), both descending
        LABFM_CUDA_TRY(ctx, cudaMemsetAsync(d_hist, 0, sizeof(unsigned int) * NBUCKET, s));
        const int nb = (int)((n + 255) / 256);
        k_bucket_count<<<nb, 256, 0, s>>>(n, order, a.row_ptr, d_hist, dmisc + 1);
        LABFM_CUDA_TRY(ctx, cudaGetLastError());
        std::vector<unsigned int> hist(NBUCKET);
        LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(hs, dmisc, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
        LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(hist.data(), d_hist, sizeof(unsigned int) * NBUCKET, cudaMemcpyDeviceToHost, s));
        LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        if (hs[1] != 0) return fail(ctx, LABFM_ERR_ARG, "order[] has entries outside 1..8");
        std::vector<unsigned int> start(NBUCKET);
        int64_t cnt[KMAX + 1] = {0}, base[KMAX + 1] = {0};
        double degsum[KMAX + 1] = {0};
        unsigned int acc = 0;
        for (int b = 0; b < NBUCKET; b++) {
            start[b] = acc;
            acc += hist[b];
            const int k = KMAX - b / 256;
            if (k >= 1) {
                if (cnt[k] == 0 && hist[b]) base[k] = start[b];
                cnt[k] += hist[b];
                degsum[k] += (double)hist[b] * (255 - b % 256);
            }
        }
        LABFM_CUDA_TRY(ctx, ctx->status_tmp.reserve(sizeof(int32_t) * (n > 0 ? n : 1)));
        int32_t *list = ctx->status_tmp.as<int32_t>();
        LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(d_cursor, start.data(), sizeof(unsigned int) * NBUCKET, cudaMemcpyHostToDevice, s));
        k_bucket_scatter<<<nb, 256, 0, s>>>(n, order, a.row_ptr, d_cursor, list);
        LABFM_CUDA_TRY(ctx, cudaGetLastError());
        // the FP64-routed orders: one persistent launch over their work items, costliest first
        OrderItems I{};
        int64_t items = 0;
        for (int k = KMAX; k >= 1; k--) {
            I.group[k] = 256;
            I.base[k] = base[k];
            I.item0[k] = items;
            if (!fp64_route(k) || !cnt[k]) continue;
            int G = 256;
            LABFM_CUDA_TRY(ctx, group_for(k, list + base[k], cnt[k], degsum[k] / (double)cnt[k], G));
            const int ng = BUILD_THREADS / G;
            I.group[k] = G;
            ctx->info_group[k] = G;
            I.cnt[k] = cnt[k];
            I.n_items[k] = (cnt[k] + ng - 1) / ng;
            items += I.n_items[k];
        }
        I.total = items;
        LABFM_CUDA_TRY(ctx, cudaMemsetAsync(dmisc, 0, sizeof(unsigned long long), s));  // the timing runs' flags
        if (items) {
            a.list = list;
            a.n_list = n;
            LABFM_CUDA_TRY(ctx, (chain ? launch_items_chain : launch_items_dw0)(a, I, ctx->num_sms, s));
        }
        // the mixed-built orders (MIXED_MIN_ORDER .. 8), highest first, each over its segment of the
        // bucketed list (one launch per order and phase: kernels shaped for each order were faster
        // than one launch per phase over all orders, which carries order 8's shared memory and
        // thread count for every node)
        for (int k = KMAX; k >= 1; k--)
            if (!fp64_route(k) && cnt[k])
                LABFM_CUDA_TRY(ctx, launch_mixed(k, list + base[k], cnt[k], degsum[k] / (double)cnt[k]));
    }
    LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(hs, dmisc, NMISC * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    if (hs[30]) return fail(ctx, LABFM_ERR_TIMEOUT, "a tensor-core completion wait gave up");
    if (mixed && hs[31]) {
        // nodes whose refinement diverged (the double-float inverse too inaccurate for the
        // iteration to contract): the FP64 build writes their weights and statuses
        const int64_t nfb = (int64_t)hs[31];
        ctx->info_fp64_rebuilt = nfb;
        a.list = ctx->mfallback.as<int32_t>();
        a.n_list = nfb;
        LABFM_CUDA_TRY(ctx, (chain ? launch_any_chain : launch_any_dw0)(a, order, uniform_order, ctx->num_sms, s));
        LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(hs, dmisc, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
        LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    }
    if (mixed)
        for (int t = 0; t < 8; t++) ctx->info_ref_hist[t] = (int64_t)hs[32 + t];
    int64_t nbad = (int64_t)hs[0];
    if (n_bad_out) *n_bad_out = nbad;
    if (nbad) return fail(ctx, LABFM_ERR_SINGULAR, std::to_string(nbad) + " node(s) flagged");
    return LABFM_OK;
}

}  // namespace labfm
