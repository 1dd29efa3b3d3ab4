// Implicit solves with the global operator matrix of Sec. 5.2 (eq. poisson_system):
//   A_ij = w^d_ji (j != i),  A_ii = -sum_j w^d_ji,   so (A x)_i = A_ii x_i + sum_j w^d_ji x_j = L^d_i(x),
// with Dirichlet rows (A_bb = 1, A_bj = 0, F_b = g_b) where the caller's mask is set, and Neumann
// ghost rows (A_gj = n_x w^x_jb + n_y w^y_jb over the stencil of the ghost's parent b, A_gb = minus
// their sum, F_g = the normal derivative at b).  The matrix is never formed: its product is a
// stencil sum over the context's CSR stencils.
//
// Solver: stabilised bi-conjugate gradients (van der Vorst, SIAM J. Sci. Stat. Comput. 13, 1992)
// with a Jacobi preconditioner M = diag(A), the preconditioned form with y = M^-1 p, z = M^-1 s:
//   rho = (r^, r); beta = (rho / rho_old)(alpha / omega); p = r + beta (p - omega v); y = M^-1 p
//   v = A y; alpha = rho / (r^, v); s = r - alpha v; z = M^-1 s; t = A z
//   omega = (t, s) / (t, t); x += alpha y + omega z; r = s - omega t
// The updates of x go to d, which is added to x when the iteration ends or starts afresh: added to x one by one, their
// roundings (of x each, a hundred times and more) would set the residual that restarts can reach, up to 1.3e-13 ||F||
// on 53^2 nodes.
// The iterations of a solve are one cooperative launch (up to ITERS_MAX of them, see GridBarrier): every block keeps its
// rows, a product is followed by a barrier, and a sum over the set rides on the barrier that its iteration needs in any
// case: each block publishes its partial sum before it and adds up all blocks' after it, in a fixed order and so to
// the same bits everywhere.  The host reads the state once per launch.  Launched as five kernels an iteration, a
// set of 66,000 nodes spent more than half of its time on launches and on the tails of the reducing blocks.
//
// The product reads the weights in the sliced layout of sell.cu: FP64 instructions bound it, one per entry there with
// one lane a node, where four lanes of a CSR row each spent as many again on combining their sums, on the diagonal and
// on the dot products as on their entries.
#include <algorithm>
#include <cmath>

#include "labfm_internal.cuh"

namespace labfm {
namespace {

constexpr int SOLVE_THREADS = 256;
constexpr int ITERS_MAX = 256;       // iterations of one launch, fewer on large sets (it holds its SMs until it ends)
constexpr int NSLOT = 8;             // partial sums: (rhat, v) | (s, s) | (t, s), (t, t) | (rhat, r), (r, r) | true residual, (b, b)

// device-resident solver state
struct SolveState {
    double rho, rho_old, alpha, omega, beta;
    double bnorm2, rnorm2, snorm2;
    double tol2;       // (tol ||b||)^2
    double resid2;     // ||b - A x||^2 at the end
    int done;          // 0 running, 1 converged, 2 breakdown, 3 iteration limit
    int skip;          // ||s|| already within the tolerance: omega = 0, d += alpha y, r = s
    int iters;
    int max_iter;
};

// The scalars of the step that follows a reduction (thread 0 of every block, on its own copy of the state):
//   step 0 (after the setup):       rnorm2, bnorm2, rho = rnorm2, alpha = omega = rho_old = 1, beta = 0
//   step 2 (after v = A y):         alpha = rho / (rhat, v)
//   step 4 (after t = A z):         skip = (s, s) <= tol2; omega = (t, s) / (t, t)
//   step 5 (after the x, r update): rho_old = rho, rho = (rhat, r), rnorm2, iters++, convergence,
//                                   beta of the next iteration
// step 4 takes s0 = (t, s), s1 = (t, t) and snorm2 as it stands.
__device__ void form_scalars(int step, double s0, double s1, SolveState *st)
{
    switch (step) {
    case 0:
        st->rnorm2 = s0;
        st->bnorm2 = s1;
        st->tol2 *= s1 > 0.0 ? s1 : 1.0;
        st->rho = s0;
        st->rho_old = st->alpha = st->omega = 1.0;
        st->beta = 0.0;
        st->iters = 0;
        st->done = (s0 <= st->tol2) ? 1 : 0;
        break;
    case 2:
        st->alpha = st->rho / s0;
        if (s0 == 0.0 || !isfinite(st->alpha)) st->done = 2;
        break;
    case 4:
        st->skip = st->snorm2 <= st->tol2 ? 1 : 0;
        st->omega = st->skip ? 0.0 : (s1 > 0.0 ? s0 / s1 : 0.0);
        if (!isfinite(st->omega)) st->done = 2;
        break;
    default:
        st->rho_old = st->rho;
        st->rho = s0;
        st->rnorm2 = s1;
        st->iters += 1;
        if (s1 <= st->tol2) st->done = 1;
        else if (st->rho == 0.0 || st->omega == 0.0 || !isfinite(s1)) st->done = 2;
        else if (st->iters >= st->max_iter) st->done = 3;
        else {
            st->beta = (st->rho / st->rho_old) * (st->alpha / st->omega);
            if (!isfinite(st->beta)) st->done = 2;
        }
        break;
    }
}

// Neumann ghost rows (Sec. 5.2): gmap[ghost[g]] = g (gmap starts at -1), with the checks the host
// reads back in flag: bit 0 an index out of range or a ghost that is its own parent, bit 1 a
// ghost listed twice, bit 2 a ghost row also marked Dirichlet, bit 3 a non-finite normal.
__global__ void k_ghost_map(int64_t n, int64_t n_ghost, const int64_t *__restrict__ ghost,
                            const int64_t *__restrict__ parent, const double *__restrict__ normal,
                            const uint8_t *__restrict__ dirichlet, int32_t *__restrict__ gmap,
                            unsigned int *__restrict__ flag)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n_ghost) return;
    const int64_t gi = ghost[g], b = parent[g];
    if (!isfinite(normal[2 * g]) || !isfinite(normal[2 * g + 1])) atomicOr(flag, 8u);
    if (gi < 0 || gi >= n || b < 0 || b >= n || gi == b) {
        atomicOr(flag, 1u);
        return;
    }
    if (dirichlet && dirichlet[gi]) atomicOr(flag, 4u);
    if (atomicCAS(&gmap[gi], -1, (int)g) != -1) atomicOr(flag, 2u);
}

// The Neumann ghost rows as the kernels read them (all null when there are none)
struct GhostRows {
    const int32_t *gmap = nullptr;   // [n]: ghost ordinal of row i, or -1
    const int64_t *parent = nullptr; // [n_ghost]
    const double *normal = nullptr;  // [n_ghost][2]
    int op_x = 0, op_y = 0;
};

// The rows in the sliced layout (a warp per slice): the weights of operator `op`, the diagonal A_ii = -sum_j w_ji, the
// Jacobi scaling 1 / A_ii, and the Dirichlet values into the initial guess: their residuals, search
// directions and updates are then exactly zero, so those entries keep f_i exactly.
// A Neumann ghost row is n_x L^(op_x) + n_y L^(op_y) at its parent b (Sec. 5.2): entry e of b's stencil gets c_e = n_x
// w^(op_x)_e + n_y w^(op_y)_e, the column of b gets -sum_e c_e (adiag), and the Jacobi scaling uses the row's true
// diagonal, the c_e of the ghost itself within b's stencil (1 if it is absent or zero).
template <class WT>
__global__ void __launch_bounds__(SOLVE_THREADS) k_solve_setup(int64_t n, SellView S, const int64_t *__restrict__ row_ptr,
                                                              const int32_t *__restrict__ col,
                                                              const WT *__restrict__ w, int n_ops, int op, GhostRows gr,
                                                              double *__restrict__ wd, double *__restrict__ dinv,
                                                              double *__restrict__ adiag,
                                                              const uint8_t *__restrict__ dirichlet,
                                                              const double *__restrict__ f, double *__restrict__ x)
{
    const SellLane l((int64_t)blockIdx.x * (SOLVE_THREADS / 32) + (threadIdx.x >> 5), threadIdx.x & 31, n, S);
    const int64_t i = l.i;
    int64_t rs = 0, re = 0;
    int g = -1;
    double nx = 0.0, ny = 0.0;
    if (i >= 0) {
        int64_t r = i;
        if (gr.gmap) g = gr.gmap[i];
        if (g >= 0) {
            r = gr.parent[g];
            nx = gr.normal[2 * g];
            ny = gr.normal[2 * g + 1];
        }
        rs = row_ptr[r];
        re = row_ptr[r + 1];
    }
    double sum = 0.0, diag = 0.0;
#pragma unroll 4
    for (int k = 0; k < l.steps; k++) {
        const int64_t e = rs + ((int64_t)k << S.lg_l) + l.h;
        double v = 0.0;
        if (e < re) {
            if (g < 0) {
                v = (double)w[e * n_ops + op];
            } else {
                v = nx * (double)w[e * n_ops + gr.op_x] + ny * (double)w[e * n_ops + gr.op_y];
                if (col[e] == i) diag += v;
            }
        }
        wd[l.at + 32 * (int64_t)k] = v;
        sum += v;
    }
    for (int o = (1 << S.lg_l) >> 1; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        diag += __shfl_xor_sync(0xffffffffu, diag, o);
    }
    if (i < 0 || l.h != 0) return;
    const bool fixed = dirichlet && dirichlet[i];
    if (fixed) x[i] = f[i];
    adiag[i] = -sum;  // A_ii (a ghost row: A_gb)
    const double a = g >= 0 ? diag : -sum;
    dinv[i] = fixed ? 1.0 : (a != 0.0 && isfinite(1.0 / a) ? 1.0 / a : 1.0);
}

struct SolveArgs {
    int64_t n;
    SellView S;
    const double *wd, *adiag, *dinv, *b;
    const uint8_t *dirichlet;
    GhostRows gr;
    double *x, *d, *r, *rhat, *p, *v, *y, *s, *z, *t;  // d: what the iteration has added to x since its start
    double *part;  // [NSLOT][blocks]
    SolveState *st;
    GridSync sync;
};

// One block's side of a run
struct SolveBlock {
    const SolveArgs &A;
    GridBarrier bar;
    int n0, n1;  // rows
    int lane, warp;
    SliceSweep<4, 1, 1, 1, true, double> sweep;

    __device__ SolveBlock(const SolveArgs &args, int64_t s0, int64_t s1)
        : A(args), bar{args.sync}, n0((int)(s0 * (32 >> args.S.lg_l))), n1((int)min(args.n, s1 * (32 >> args.S.lg_l))),
          lane(threadIdx.x & 31), warp(threadIdx.x >> 5)
    {
        sweep.place(A.n, A.S);
        sweep.preload(A.n, A.S, A.wd);
    }

    // A x over the block's rows with the matrix in its global form (Sec. 5.2), A_ii x_i + sum_j w_ji x_j, one FP64
    // multiply-add per stencil entry (Dirichlet rows: x_i; a Neumann ghost row: the stencil of its parent b with the
    // ghost weights, and the diagonal term on x_b): fn(i, (A x)_i, own_i) on one lane per row, own_i read ahead.  The first
    // steps of the next product are on their way when it returns.
    // DIFFERENCES: as sum_j w_ji (x_j - x_i), for true residuals.  The terms of the global form cancel (by a factor of
    // about (L / h)^2 in a Laplacian of a smooth x), and its roundings, 1e-13 ||F|| on 41^2 nodes, made solves to that
    // tolerance end or fail by the order of the sums; the differences hardly cancel.
    template <bool DIFFERENCES, class Fn>
    __device__ __forceinline__ void product(const double *x, const double *own, Fn fn)
    {
        struct Row {
            double xi, ai, oi, sum[2];
            bool row, fixed;
        };
        sweep.run(
            A.n, A.S, A.wd,
            [&](const SellLane &l, bool mine) {
                Row v;
                v.xi = v.ai = v.oi = v.sum[0] = v.sum[1] = 0.0;
                v.fixed = false;
                v.row = mine && l.i >= 0 && l.h == 0;
                if (v.row || (DIFFERENCES && l.i >= 0)) {
                    int64_t src = l.i;
                    if (A.gr.gmap && A.gr.gmap[l.i] >= 0) src = A.gr.parent[A.gr.gmap[l.i]];
                    v.xi = x[src];
                }
                if (v.row) {
                    v.oi = own[l.i];
                    if (!DIFFERENCES) v.ai = A.adiag[l.i];
                    v.fixed = A.dirichlet && A.dirichlet[l.i];
                }
                return v;
            },
            [&](int j, double(&xv)[1]) { xv[0] = x[j]; },
            [&](Row &v, int q, const double(&xv)[1], const double(&w)[1]) {
                v.sum[q & 1] = fma(DIFFERENCES ? xv[0] - v.xi : xv[0], w[0], v.sum[q & 1]);
            },
            [&](const Row &v, double(&p)[1]) { p[0] = v.sum[0] + v.sum[1]; },
            [&](const SellLane &l, const Row &v, const double(&p)[1]) {
                double acc = p[0];
                for (int o = (1 << A.S.lg_l) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (v.row) fn(l.i, v.fixed ? v.xi : DIFFERENCES ? acc : fma(v.ai, v.xi, acc), v.oi);
            });
        sweep.place(A.n, A.S);
        sweep.preload(A.n, A.S, A.wd);
    }

    // The sums of a and b over all blocks (NQ = 1: of a) through partial sums in slots q0 and q0 + 1, around a barrier; on
    // thread 0 in out.  false: the barrier gave up.  Four warps add up a block's values, one from each of the SM's
    // quarters: a shuffle tree in all sixteen would take the FP64 pipe longer.
    template <int NQ>
    __device__ bool reduce(int q0, double a, double b, double (&out)[2])
    {
        __shared__ double sh[NQ][RUN_THREADS], quarter[NQ][4], total[NQ];
        __syncthreads();
        sh[0][threadIdx.x] = a;
        if (NQ > 1) sh[NQ - 1][threadIdx.x] = b;
        __syncthreads();
        if (warp < 4 * NQ) {
            const double *v = sh[warp >> 2] + 128 * (warp & 3) + lane;
            double w = (v[0] + v[32]) + (v[64] + v[96]);
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) quarter[warp >> 2][warp & 3] = w;
        }
        __syncthreads();
        if (threadIdx.x < NQ) {
            const double *q = quarter[threadIdx.x];
            A.part[(q0 + threadIdx.x) * gridDim.x + blockIdx.x] = (q[0] + q[1]) + (q[2] + q[3]);
        }
        if (!bar.wait()) return false;
        if (warp < NQ) {
            const double *p = A.part + (q0 + warp) * gridDim.x;
            double w0 = 0.0, w1 = 0.0;
            for (unsigned k = lane; k < gridDim.x; k += 64) {
                w0 += __ldcg(p + k);
                if (k + 32 < gridDim.x) w1 += __ldcg(p + k + 32);
            }
            double w = w0 + w1;
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) total[warp] = w;
        }
        __syncthreads();
        out[0] = total[0];
        out[1] = total[NQ - 1];
        return true;
    }
};

// Up to `most` iterations; with `start` first the residual and the starting scalars of the iterate in x.  Once the
// iteration has ended, the true residual of x too.  257^2 nodes, 49 entries each: 33 to 38 us an iteration (56 to 62 as five
// launches), 12 of them the products' FP64 issue, 8 the five barriers, the rest latency between them.
__global__ void __launch_bounds__(RUN_THREADS, 1) k_solve_run(SolveArgs A, int start, int most)
{
    __shared__ SolveState st;
    int64_t s0, s1;
    block_share(A.S, s0, s1);
    GridBarrier{A.sync}.check();
    share_out(A.S, s0, s1);
    if (GridBarrier::stopped()) {
        if (threadIdx.x == 0) *(volatile unsigned *)A.sync.gave_up = 1u;  // the host learns that no iteration was made
        return;
    }
    SolveBlock B(A, s0, s1);
    if (threadIdx.x == 0) st = *A.st;
    __syncthreads();
    double sum[2] = {0.0, 0.0};
    auto scalars = [&](int step) {
        if (threadIdx.x == 0) form_scalars(step, sum[0], sum[1], &st);
        __syncthreads();
    };
    if (start) {
        double rr = 0.0, bb = 0.0;
        B.product<true>(A.x, A.b, [&](int64_t i, double ax, double bi) {
            const double ri = bi - ax;
            A.d[i] = 0.0;
            A.r[i] = ri;
            A.rhat[i] = ri;
            A.p[i] = 0.0;
            A.v[i] = 0.0;
            rr = fma(ri, ri, rr);
            bb = fma(bi, bi, bb);
        });
        if (!B.reduce<2>(4, rr, bb, sum)) return;
        scalars(0);
    }
    for (int it = 0; it < most && !st.done; it++) {
        // p = r + beta (p - omega v); y = dinv p
        {
            const double beta = st.beta, omega = st.omega;
            for (int i = B.n0 + threadIdx.x; i < B.n1; i += RUN_THREADS) {
                const double pi = fma(beta, fma(-omega, A.v[i], A.p[i]), A.r[i]);
                A.p[i] = pi;
                A.y[i] = A.dinv[i] * pi;
            }
        }
        if (!B.bar.wait()) return;
        // v = A y, (rhat, v) -> alpha
        double d0 = 0.0, d1 = 0.0;
        B.product<false>(A.y, A.rhat, [&](int64_t i, double vi, double hi) {
            A.v[i] = vi;
            d0 = fma(hi, vi, d0);
        });
        if (!B.reduce<1>(0, d0, 0.0, sum)) return;
        scalars(2);
        if (st.done) break;
        // s = r - alpha v; z = dinv s; (s, s)
        d0 = 0.0;
        {
            const double alpha = st.alpha;
            for (int i = B.n0 + threadIdx.x; i < B.n1; i += RUN_THREADS) {
                const double si = fma(-alpha, A.v[i], A.r[i]);
                A.s[i] = si;
                A.z[i] = A.dinv[i] * si;
                d0 = fma(si, si, d0);
            }
        }
        if (!B.reduce<1>(1, d0, 0.0, sum)) return;
        if (threadIdx.x == 0) st.snorm2 = sum[0];
        // t = A z, (t, s), (t, t) -> omega
        d0 = 0.0;
        B.product<false>(A.z, A.s, [&](int64_t i, double ti, double si) {
            A.t[i] = ti;
            d0 = fma(si, ti, d0);
            d1 = fma(ti, ti, d1);
        });
        if (!B.reduce<2>(2, d0, d1, sum)) return;
        scalars(4);
        if (st.done) break;
        // d += alpha y + omega z; r = s - omega t; (rhat, r), (r, r) -> rho, beta, convergence
        d0 = d1 = 0.0;
        {
            const double alpha = st.alpha, omega = st.omega;
            for (int i = B.n0 + threadIdx.x; i < B.n1; i += RUN_THREADS) {
                A.d[i] = fma(omega, A.z[i], fma(alpha, A.y[i], A.d[i]));
                const double ri = fma(-omega, A.t[i], A.s[i]);
                A.r[i] = ri;
                d0 = fma(A.rhat[i], ri, d0);
                d1 = fma(ri, ri, d1);
            }
        }
        if (!B.reduce<2>(4, d0, d1, sum)) return;
        scalars(5);
    }
    if (st.done) {
        for (int i = B.n0 + threadIdx.x; i < B.n1; i += RUN_THREADS) A.x[i] += A.d[i];
        if (!B.bar.wait()) return;
        double rr = 0.0, bb = 0.0;
        B.product<true>(A.x, A.b, [&](int64_t, double ax, double bi) {
            const double ri = bi - ax;
            rr = fma(ri, ri, rr);
            bb = fma(bi, bi, bb);
        });
        if (!B.reduce<2>(6, rr, bb, sum)) return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (st.done) {
            st.resid2 = sum[0];
            st.bnorm2 = sum[1];
        }
        *A.st = st;
    }
}

}  // namespace

labfm_status run_solve(labfm_ctx *ctx, int op, const double *f, double *phi, const uint8_t *dirichlet,
                       const SolveNeumann &nm, double tol, int max_iter, int *iters_out, double *resid_out)
{
    cudaStream_t s = ctx->stream;
    const int64_t n = ctx->n, nnz = ctx->nnz;
    // Neumann ghost rows: map and checks, read back with one synchronisation
    GhostRows gr;
    if (nm.n_ghost > 0) {
        const int64_t ng = nm.n_ghost;
        const size_t map_bytes = ((sizeof(int32_t) * (size_t)n + 15) / 16) * 16;
        LABFM_CUDA_TRY(ctx, ctx->sol_gmap.reserve(map_bytes + 16));
        int32_t *gmap = ctx->sol_gmap.as<int32_t>();
        unsigned int *gflag = reinterpret_cast<unsigned int *>(reinterpret_cast<char *>(gmap) + map_bytes);
        LABFM_CUDA_TRY(ctx, cudaMemsetAsync(gmap, 0xff, sizeof(int32_t) * (size_t)n, s));  // -1
        LABFM_CUDA_TRY(ctx, cudaMemsetAsync(gflag, 0, sizeof(unsigned int), s));
        k_ghost_map<<<(unsigned)((ng + 255) / 256), 256, 0, s>>>(n, ng, nm.ghost, nm.parent, nm.normal, dirichlet,
                                                                 gmap, gflag);
        LABFM_CUDA_TRY(ctx, cudaGetLastError());
        unsigned int *hs = (unsigned int *)ctx->host_small;
        LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(hs, gflag, sizeof(unsigned int), cudaMemcpyDeviceToHost, s));
        LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        const unsigned flag = *hs;
        if (flag & 1u) return fail(ctx, LABFM_ERR_ARG, "a ghost or parent index is out of range, or a ghost is its own parent");
        if (flag & 2u) return fail(ctx, LABFM_ERR_ARG, "a ghost row is listed twice");
        if (flag & 4u) return fail(ctx, LABFM_ERR_ARG, "a ghost row is also a Dirichlet row");
        if (flag & 8u) return fail(ctx, LABFM_ERR_ARG, "a ghost normal is not finite");
        gr.gmap = gmap;
        gr.parent = nm.parent;
        gr.normal = nm.normal;
        gr.op_x = nm.op_x;
        gr.op_y = nm.op_y;
    }
    // the layout: the stencils' own, or with ghost rows one of this call
    Sell &L = gr.gmap ? ctx->sell_ghost : ctx->sell;
    const labfm_status ls = gr.gmap ? build_sell(ctx, L, gr.gmap, gr.parent) : ensure_sell(ctx);
    if (ls != LABFM_OK) return ls;
    const SellView S = sell_view(L);
    LABFM_CUDA_TRY(ctx, ctx->sol_w.reserve(sizeof(double) * (L.places > 0 ? L.places : 1)));
    LABFM_CUDA_TRY(ctx, ctx->sol_vec.reserve(sizeof(double) * 11 * n));
    LABFM_CUDA_TRY(ctx, ctx->sol_part.reserve(sizeof(double) * NSLOT * (size_t)ctx->num_sms + sizeof(SolveState)));
    LABFM_CUDA_TRY(ctx, ensure_sync(ctx));
    double *V = ctx->sol_vec.as<double>();
    double *dinv = V, *r = V + n, *rhat = V + 2 * n, *p = V + 3 * n, *v = V + 4 * n, *y = V + 5 * n, *sv = V + 6 * n,
           *z = V + 7 * n, *t = V + 8 * n, *adiag = V + 9 * n, *d = V + 10 * n;
    double *part = ctx->sol_part.as<double>();
    SolveState *st = reinterpret_cast<SolveState *>(part + NSLOT * (size_t)ctx->num_sms);
    const double *wd = ctx->sol_w.as<double>();
    {
        const unsigned blocks = (unsigned)((S.n_slices + SOLVE_THREADS / 32 - 1) / (SOLVE_THREADS / 32));
        const int64_t *rp = ctx->row_ptr.as<int64_t>();
        const int32_t *cl = ctx->col.as<int32_t>();
        if (ctx->wdtype == LABFM_F64)
            k_solve_setup<double><<<blocks, SOLVE_THREADS, 0, s>>>(n, S, rp, cl, ctx->w.as<double>(), ctx->n_ops, op, gr,
                                                                  ctx->sol_w.as<double>(), dinv, adiag, dirichlet, f, phi);
        else
            k_solve_setup<float><<<blocks, SOLVE_THREADS, 0, s>>>(n, S, rp, cl, ctx->w.as<float>(), ctx->n_ops, op, gr,
                                                                 ctx->sol_w.as<double>(), dinv, adiag, dirichlet, f, phi);
        LABFM_CUDA_TRY(ctx, cudaGetLastError());
    }
    SolveState init{};
    init.tol2 = tol * tol;
    init.max_iter = max_iter;
    LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(st, &init, sizeof(SolveState), cudaMemcpyHostToDevice, s));
    const SolveArgs args{n, S, wd, adiag, dinv, f, dirichlet, gr, phi, d, r, rhat, p, v, y, sv, z, t, part, st, grid_sync(ctx, LABFM_SOLVE_GAVE_UP)};
    const int most = (int)std::max<int64_t>(8, std::min<int64_t>(ITERS_MAX, (int64_t)1000000000 / (nnz + 100000)));
    // Launches until the state says that the iteration ended, with the true residual.  BiCGStab
    // restarts from the current iterate (r = F - A Phi, r^ = r), at most MAX_RESTARTS times
    // within max_iter in total, in two cases: the recurrence residual, which drifts from the
    // true one in finite precision, says converged while the true residual is above tol; or the
    // iteration broke down (rho = (r^, r), (r^, v) or omega vanished or was not finite) with a
    // finite iterate.  The second is the usual remedy for a breakdown: the shadow residual r^
    // has become orthogonal to the Krylov space, and a fresh r^ = r starts a new one.  (No
    // launch after the one that flagged the breakdown updates Phi, except when the residual
    // norm itself was not finite, which the finite-residual condition excludes.)
    constexpr int MAX_RESTARTS = 8;
    SolveState h{};
    int total = 0, restarts = 0;
    double resid = 0.0;
    cudaError_t le = cudaSuccess;
    int start = 1;
    while (true) {
        do {
            le = launch_run(ctx, S, k_solve_run, args, start, most);
            start = 0;
            if (le == cudaSuccess) le = cudaMemcpyAsync(&h, st, sizeof(SolveState), cudaMemcpyDeviceToHost, s);
            if (le == cudaSuccess) le = cudaStreamSynchronize(s);
            if (le != cudaSuccess) return cuda_fail(ctx, le, "BiCGStab iterations");
            const bool mine = gave_up(ctx, LABFM_SOLVE_GAVE_UP);
            if (const labfm_status rs = run_gave_up(ctx)) return rs;
            if (mine) return fail(ctx, LABFM_ERR_TIMEOUT, "a wait between the solver's blocks gave up");
        } while (!h.done);
        total += h.iters;
        resid = std::sqrt(h.resid2) / (h.bnorm2 > 0.0 ? std::sqrt(h.bnorm2) : 1.0);
        const bool drifted = h.done == 1 && resid > tol, broke_down = h.done == 2;
        if ((drifted || broke_down) && std::isfinite(resid) && restarts < MAX_RESTARTS && total < max_iter) {
            restarts++;
            init.max_iter = max_iter - total;
            LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(st, &init, sizeof(SolveState), cudaMemcpyHostToDevice, s));
            start = 1;
            continue;
        }
        break;
    }
    if (iters_out) *iters_out = total;
    if (resid_out) *resid_out = resid;
    if (h.done == 1 && std::isfinite(resid) && resid <= tol) return LABFM_OK;
    return fail(ctx, LABFM_ERR_NOT_CONVERGED,
                h.done == 2   ? "BiCGStab breakdown (rho, alpha or omega vanished or was not finite)"
                : h.done == 1 ? "the true residual stayed above tol after the restarts"
                              : "BiCGStab did not reach the tolerance within max_iter iterations");
}

}  // namespace labfm
