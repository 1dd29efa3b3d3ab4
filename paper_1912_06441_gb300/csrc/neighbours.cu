// Stencil search (Sec. 2: all j != i with |r_ji| < 2 h_i) on a uniform cell grid.
//
// Cells have side >= 2 h_max, so every neighbour of a node lies in its own cell or one of
// the 8 cells around it (with wrap-around in a periodic box).  Nodes are counting-sorted by
// cell; a warp counts the neighbours of a few nodes in cell order, which share their candidates, a prefix sum gives
// the CSR row pointers, and a second sweep collects each row in shared memory, sorts it in registers and writes it
// whole.  The distance test is evaluated in IEEE double
// with explicitly rounded operations (no fused multiply-add), so the result does not depend
// on the compiler's contraction choices; a float pre-classification with a proven error bound
// settles every candidate that is not within a thin shell at the radius (on GB300 the double
// test costs FP64-pipe time per candidate), and the shell goes to the double test, so the
// stencils are those of the double test bit for bit.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "labfm_internal.cuh"

namespace labfm {
namespace {

constexpr int NB_THREADS = 256;
constexpr int ROW_MAX = 128;  // entries of a row that a warp sorts in registers

struct Grid {
    double lo[2], L[2], halfL[2], inv_cs[2];
    int nc[2];
    int periodic;
    // float pre-filter of the distance test: box sides and half
    // sides in float, the bound E on |dx_float - dx| (roundings of the coordinates, the
    // difference and the wrap), and the largest (2h)^2 for which the float wrap cannot differ
    // from the double one on a candidate near the radius
    float Lf[2], halfLf[2];
    float E;
    double r2_wrap_max;
};

__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }

// Validate nodes and find max h.  misc[0] = bits of max h, misc[1] = number of bad nodes.  The context's copies of
// the positions and h are written on the way (xy_out, h_out; null: no copies).
__global__ void k_check(int64_t n, const double *__restrict__ xy, const double *__restrict__ h, double lo0, double lo1,
                        double hi0, double hi1, unsigned long long *__restrict__ misc, double2 *__restrict__ xy_out,
                        double *__restrict__ h_out)
{
    __shared__ unsigned long long s_max[NB_THREADS / 32];
    __shared__ unsigned int s_bad[NB_THREADS / 32];
    unsigned long long mx = 0;
    unsigned int bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double x = xy[2 * i], y = xy[2 * i + 1], hv = h[i];
        if (xy_out) {
            xy_out[i] = make_double2(x, y);
            h_out[i] = hv;
        }
        bool ok = isfinite(x) && isfinite(y) && isfinite(hv) && hv > 0.0 && x >= lo0 && x <= hi0 && y >= lo1 &&
                  y <= hi1;
        if (!ok) bad++;
        else mx = max(mx, dbits(hv));  // positive doubles order like their bit patterns
    }
    for (int o = 16; o > 0; o >>= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        bad += __shfl_xor_sync(0xffffffffu, bad, o);
    }
    int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_max[w] = mx;
        s_bad[w] = bad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int t = 1; t < NB_THREADS / 32; t++) {
            mx = max(mx, s_max[t]);
            bad += s_bad[t];
        }
        atomicMax(&misc[0], mx);
        if (bad) atomicAdd(&misc[1], (unsigned long long)bad);
    }
}

__device__ __forceinline__ int cell_coord(double x, double lo, double inv_cs, int nc)
{
    double t = __dmul_rn(__dsub_rn(x, lo), inv_cs);
    int c = (int)floor(t);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

__global__ void k_cell_assign(int64_t n, const double *__restrict__ xy, Grid g, int32_t *__restrict__ cell_of,
                              int32_t *__restrict__ cell_count, int32_t *__restrict__ rank, int64_t *__restrict__ longest)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && longest) *longest = 0;  // until the rows' offsets are formed
    if (i >= n) return;
    int cx = cell_coord(xy[2 * i], g.lo[0], g.inv_cs[0], g.nc[0]);
    int cy = cell_coord(xy[2 * i + 1], g.lo[1], g.inv_cs[1], g.nc[1]);
    int c = cy * g.nc[0] + cx;
    cell_of[i] = c;
    rank[i] = atomicAdd(&cell_count[c], 1);  // the node's place within its cell
}

__global__ void k_cell_scatter(int64_t n, const double *__restrict__ xy, const int32_t *__restrict__ cell_of,
                               const int64_t *__restrict__ cell_start, const int32_t *__restrict__ rank,
                               int32_t *__restrict__ cell_nodes, double2 *__restrict__ cell_xy,
                               float2 *__restrict__ cell_xyf)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int c = cell_of[i];
    int64_t pos = cell_start[c] + rank[i];
    cell_nodes[pos] = (int32_t)i;
    const double x = xy[2 * i], y = xy[2 * i + 1];
    cell_xy[pos] = make_double2(x, y);
    if (cell_xyf) cell_xyf[pos] = make_float2((float)x, (float)y);
}

// The up-to-3 distinct cell coordinates around c along one axis.
__device__ __forceinline__ int axis_cells(int c, int nc, int periodic, int out[3])
{
    int m = 0;
    for (int d = -1; d <= 1; d++) {
        int v = c + d;
        if (periodic) {
            v = v < 0 ? v + nc : (v >= nc ? v - nc : v);
        } else if (v < 0 || v >= nc) {
            continue;
        }
        bool dup = false;
        for (int t = 0; t < m; t++) dup |= (out[t] == v);
        if (!dup) out[m++] = v;
    }
    return m;
}

// The exact distance test of Sec. 2 in IEEE double, explicitly rounded (no contraction).
__device__ __forceinline__ bool within_exact(double qx, double qy, double xi, double yi, double R2, const Grid &g)
{
    double dx = __dsub_rn(qx, xi);
    double dy = __dsub_rn(qy, yi);
    if (g.periodic) {
        if (dx > g.halfL[0]) dx = __dsub_rn(dx, g.L[0]);
        else if (dx < -g.halfL[0]) dx = __dadd_rn(dx, g.L[0]);
        if (dy > g.halfL[1]) dy = __dsub_rn(dy, g.L[1]);
        else if (dy < -g.halfL[1]) dy = __dadd_rn(dy, g.L[1]);
    }
    double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    return r2 < R2;
}

// Ascending sort of a warp's row of cnt <= 32 E entries from shared memory, element e 32 + lane in register e of
// lane (a bitonic network; exchanges of partners 32 or more apart stay within a lane), then the row to out.
template <int E>
__device__ __forceinline__ void sort_row(const int32_t *buf, int cnt, int lane, int32_t *__restrict__ out)
{
    int v[E];
#pragma unroll
    for (int e = 0; e < E; e++) v[e] = 32 * e + lane < cnt ? buf[32 * e + lane] : 0x7fffffff;
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int e = 0; e < E; e++) {
                    const int f = e ^ (j / 32);
                    if (f > e) {
                        const bool up = ((32 * e) & k) == 0;  // k > 32 here, or all of them up at the last k
                        const int a = min(v[e], v[f]), b = max(v[e], v[f]);
                        v[e] = up ? a : b;
                        v[f] = up ? b : a;
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; e++) {
                    const int o = __shfl_xor_sync(0xffffffffu, v[e], j);
                    const bool up = ((32 * e + lane) & k) == 0;
                    v[e] = (((lane & j) == 0) == up) ? min(v[e], o) : max(v[e], o);
                }
            }
        }
    }
#pragma unroll
    for (int e = 0; e < E; e++)
        if (32 * e + lane < cnt) out[32 * e + lane] = v[e];
}

// Ascending sort of a longer row in place in global memory by one warp: the bitonic network whose exchanges all
// put the smaller entry first, so that entries from cnt on may be taken as larger than any and left out.
__device__ __noinline__ void sort_long_row(int32_t *row, int cnt, int lane)
{
    for (int64_t k = 2; (k >> 1) < cnt; k <<= 1) {
        for (int64_t j = k >> 1; j > 0; j >>= 1) {
            __syncwarp();
            const int64_t flip = j == (k >> 1) ? k - 1 : j;
            for (int64_t a = lane; a < cnt; a += 32) {
                const int64_t b = a ^ flip;
                if (b > a && b < cnt && row[a] > row[b]) {
                    const int32_t t = row[a];
                    row[a] = row[b];
                    row[b] = t;
                }
            }
        }
    }
}

// The float pre-filter of the distance test.  r2f, the squared distance from the float coordinates, differs from the double
// r2 by at most D = 2E s + 2E^2 + 2^-23 r2f, s = |dx_f| + |dy_f| (E bounds the error of dx_f and dy_f); a candidate with
// r2f below or above (2h)^2 by more than 2D + 2^-22 (2h)^2 is decided (the second half of it and the last term are
// more than the roundings of this test itself), and only the rest (a thin shell at the radius) takes the double test.
// The result is the double test's, bit for bit; on GB300 the double test costs FP64-pipe time per candidate, the
// float one does not.
struct Prefilter {
    float xi, yi, below, above;  // (2h)^2 less and plus the terms that no candidate changes
    __device__ __forceinline__ Prefilter(float x, float y, float R2f, const Grid &g) : xi(x), yi(y)
    {
        const float m = 2.3841858e-7f * R2f + 4.0f * g.E * g.E;
        below = R2f - m;
        above = R2f + m;
    }
    __device__ __forceinline__ void test(float2 q, bool wrap, const Grid &g, bool &in, bool &out) const
    {
        float dx = q.x - xi, dy = q.y - yi;
        if (wrap) {
            if (dx > g.halfLf[0]) dx -= g.Lf[0];
            else if (dx < -g.halfLf[0]) dx += g.Lf[0];
            if (dy > g.halfLf[1]) dy -= g.Lf[1];
            else if (dy < -g.halfLf[1]) dy += g.Lf[1];
        }
        const float r2 = fmaf(dx, dx, dy * dy);
        const float t = (4.0f * g.E) * (fabsf(dx) + fabsf(dy));
        in = fmaf(r2, 1.0f + 2.3841858e-7f, t) < below;
        out = fmaf(r2, 1.0f - 2.3841858e-7f, -t) > above;
    }
};

// The candidates of a cell: the up to nine cells around it.  The cells of a row lie one behind another in cell order, so
// they are three runs of nodes, and three more where the row wraps around; q = 0 .. total - 1 numbers them.
struct Candidates {
    int s[6], e[6];  // run k: candidates up to e[k] are node s[k] + q in cell order
    int total;
    bool wrap;       // an offset may have to be wrapped (a periodic box, the cell at its edge or fewer than five cells a side)
    __device__ __forceinline__ Candidates(int c, const Grid &g, const int64_t *__restrict__ cell_start)
    {
        const int nx = g.nc[0], cx = c % nx, cy = c / nx;
        // the x range of cells, [xa, xb], and behind it the wrapped one [xc, xc] if there is one (xc < 0: none)
        int xa = cx - 1, xb = cx + 1, xc = -1;
        if (g.periodic && nx > 3) {
            if (xa < 0) xc = nx - 1;
            if (xb >= nx) xc = 0;
        } else if (g.periodic) {
            xa = 0;
            xb = nx - 1;
        }
        xa = max(xa, 0);
        xb = min(xb, nx - 1);
        // the distinct cell rows around cy
        const int ny = g.nc[1];
        int y0 = cy - 1, y1 = cy, y2 = cy + 1, my = 3;
        if (g.periodic) {
            if (y0 < 0) y0 += ny;
            if (y2 >= ny) y2 -= ny;
            my = ny < 3 ? ny : 3;
            if (ny < 3) {
                y0 = 0;
                y1 = 1;
            }
        } else {
            if (y2 >= ny) my = 2;
            if (y0 < 0) {
                y0 = y1;
                y1 = y2;
                my--;
            }
        }
        wrap = g.periodic && (nx < 5 || g.nc[1] < 5 || xc >= 0 || cy == 0 || cy == g.nc[1] - 1);
        total = 0;
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const int a = k % 3;
            int from = 0, len = 0;
            if (a < my && (k < 3 || xc >= 0)) {
                const int64_t row = (int64_t)(a == 0 ? y0 : a == 1 ? y1 : y2) * nx;
                from = (int)cell_start[row + (k < 3 ? xa : xc)];
                len = (int)cell_start[row + (k < 3 ? xb : xc) + 1] - from;
            }
            s[k] = from - total;
            total += len;
            e[k] = total;
        }
    }
    __device__ __forceinline__ int place(int q) const  // in cell order
    {
        int p = s[0];
        p = q >= e[0] ? s[1] : p;
        p = q >= e[1] ? s[2] : p;
        if (e[5] > e[2]) {
            p = q >= e[2] ? s[3] : p;
            p = q >= e[3] ? s[4] : p;
            p = q >= e[4] ? s[5] : p;
        }
        return p + q;
    }
};

// Float coordinates of the node at p in cell order, from the float copy, or where there is none (the search on a fixed
// scratch array) the same values converted again: 360^2 nodes at order 4 in 224 us, 838 with the double test alone.  (The
// sweeps test the copy against null although it is there: left out, the search took 2 to 3 % longer.)
template <bool COPY>
__device__ __forceinline__ float2 float_at(int64_t p, const double2 *__restrict__ cell_xy, const float2 *__restrict__ cell_xyf)
{
    if (COPY) return cell_xyf[p];
    const double2 q = cell_xy[p];
    return make_float2((float)q.x, (float)q.y);
}

// One sweep over the candidates of every node; WRITE = false: count; true: write col[].  A warp takes SWEEP_NODES
// consecutive nodes in cell order.  The nodes of a cell share their candidates, which the warp keeps in registers (up to
// SWEEP_REGS per lane; more are read again for every node): per node there is the test of each candidate, a ballot
// that gives the hits' places in the row, and the sort.  (A warp per node spent most of its time finding the
// node's cells: 180 us a count and 254 us a write at 512^2, order 8, against 124 and 185 now; a thread per node took 102
// and 817.)
constexpr int SWEEP_NODES = 8;
constexpr int SWEEP_REGS = 8;
template <bool WRITE, bool COPY>
__global__ void __launch_bounds__(NB_THREADS) k_sweep(int64_t n, const double *__restrict__ h, Grid g,
                                                      const int32_t *__restrict__ cell_of,
                                                      const int64_t *__restrict__ cell_start,
                                                      const int32_t *__restrict__ cell_nodes,
                                                      const double2 *__restrict__ cell_xy,
                                                      const float2 *__restrict__ cell_xyf, int32_t *__restrict__ counts,
                                                      const int64_t *__restrict__ row_ptr, int32_t *__restrict__ col)
{
    __shared__ int32_t s_row[WRITE ? NB_THREADS / 32 : 1][WRITE ? ROW_MAX : 1];
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t t0 = ((int64_t)blockIdx.x * (NB_THREADS / 32) + (threadIdx.x >> 5)) * SWEEP_NODES;
    if (t0 >= n) return;  // whole warps
    const int nodes = (int)min((int64_t)SWEEP_NODES, n - t0);
    // lane k: node k of the warp
    int my_i = 0, my_cell = -1, my_total = 0, my_cnt = 0;
    int64_t my_base = 0;
    double2 my_at = make_double2(0.0, 0.0);
    double my_R2 = 0.0;
    if (lane < nodes) {
        my_i = cell_nodes[t0 + lane];
        my_at = cell_xy[t0 + lane];
        const double R = 2.0 * h[my_i];
        my_R2 = __dmul_rn(R, R);
        my_cell = cell_of[my_i];
        if (WRITE) {
            my_base = row_ptr[my_i];
            my_total = (int)(row_ptr[my_i + 1] - my_base);
        }
    }
    const float my_xf = (float)my_at.x, my_yf = (float)my_at.y, my_R2f = (float)my_R2;
    // float classification only where the float wrap cannot flip a candidate near the radius
    const int my_filt = (!COPY || cell_xyf != nullptr) && (!g.periodic || my_R2 <= g.r2_wrap_max);
    for (int k0 = 0; k0 < nodes;) {
        const int c = __shfl_sync(all, my_cell, k0);
        const Candidates cand(c, g, cell_start);
        float2 cq[SWEEP_REGS];
        int cj[SWEEP_REGS];
        unsigned valid = 0;
        auto load = [&](int c0) {
            valid = 0;
#pragma unroll
            for (int r = 0; r < SWEEP_REGS; r++) {
                const int q = c0 + 32 * r + lane;
                cq[r] = make_float2(0.0f, 0.0f);
                cj[r] = 0;
                if (q < cand.total) {
                    const int p = cand.place(q);
                    cj[r] = cell_nodes[p];
                    if (!COPY || cell_xyf) cq[r] = float_at<COPY>(p, cell_xy, cell_xyf);
                    valid |= 1u << r;
                }
            }
        };
        const bool kept = cand.total <= 32 * SWEEP_REGS;
        if (kept) load(0);
        // this cell's nodes among the warp's
        const unsigned same = __ballot_sync(all, lane >= k0 && my_cell == c);
        const int k1 = 32 - __clz(same);  // cell order: consecutive
        for (int k = k0; k < k1; k++) {
            const int i = __shfl_sync(all, my_i, k);
            const Prefilter pre(__shfl_sync(all, my_xf, k), __shfl_sync(all, my_yf, k), __shfl_sync(all, my_R2f, k), g);
            const bool filt = __shfl_sync(all, my_filt, k) != 0;
            const int64_t base = WRITE ? __shfl_sync(all, my_base, k) : 0;
            int32_t *dst = nullptr;
            if constexpr (WRITE) dst = __shfl_sync(all, my_total, k) <= ROW_MAX ? s_row[threadIdx.x >> 5] : col + base;
            int cnt = 0;
            for (int c0 = 0; c0 < cand.total; c0 += 32 * SWEEP_REGS) {
                if (!kept) load(c0);
                unsigned hit = 0, open = 0;  // bit r: candidate 32 r + lane is inside, is to take the double test
#pragma unroll
                for (int r = 0; r < SWEEP_REGS; r++)
                    if (c0 + 32 * r < cand.total) {
                        bool in, out;
                        pre.test(cq[r], cand.wrap, g, in, out);
                        if (cj[r] != i) {
                            if (in) hit |= 1u << r;
                            else if (!out) open |= 1u << r;
                        }
                        if (!filt && cj[r] != i) open |= 1u << r;
                    }
                hit = filt ? hit & valid : 0u;
                open &= valid;
                if (__any_sync(all, open != 0)) {
                    const double xd = __shfl_sync(all, my_at.x, k), yd = __shfl_sync(all, my_at.y, k);
                    const double R2 = __shfl_sync(all, my_R2, k);
                    while (open) {
                        const int r = __ffs(open) - 1;
                        open &= open - 1;
                        const double2 qd = cell_xy[cand.place(c0 + 32 * r + lane)];
                        if (within_exact(qd.x, qd.y, xd, yd, R2, g)) hit |= 1u << r;
                    }
                }
                if constexpr (WRITE) {
                    __syncwarp();
#pragma unroll
                    for (int r = 0; r < SWEEP_REGS; r++)
                        if (c0 + 32 * r < cand.total) {
                            const bool in = (hit >> r) & 1u;
                            const unsigned hits = __ballot_sync(all, in);
                            if (in) dst[cnt + __popc(hits & ((1u << lane) - 1u))] = cj[r];
                            cnt += __popc(hits);
                        }
                } else {
                    cnt += (int)__reduce_add_sync(all, (unsigned)__popc(hit));
                }
            }
            if constexpr (!WRITE) {
                if (lane == k) my_cnt = cnt;
            } else {
                __syncwarp();
                if (cnt <= 32) sort_row<1>(dst, cnt, lane, col + base);
                else if (cnt <= 64) sort_row<2>(dst, cnt, lane, col + base);
                else if (cnt <= ROW_MAX) sort_row<4>(dst, cnt, lane, col + base);
                else sort_long_row(col + base, cnt, lane);
                __syncwarp();  // the row is read before the next one is collected
            }
        }
        k0 = k1;
    }
    if (!WRITE && lane < nodes) counts[my_i] = my_cnt;
}

// The same with a thread per node, in cell order, its row sorted by insertion: for large sets of few nodes to a cell, where
// the rows are short and a warp's eight nodes lie in several cells.
template <bool WRITE, bool COPY>
__global__ void k_sweep_sparse(int64_t n, const double *__restrict__ h, Grid g,
                        const int32_t *__restrict__ cell_of, const int64_t *__restrict__ cell_start,
                        const int32_t *__restrict__ cell_nodes, const double2 *__restrict__ cell_xy,
                        const float2 *__restrict__ cell_xyf, int32_t *__restrict__ counts,
                        const int64_t *__restrict__ row_ptr, int32_t *__restrict__ col)
{
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    int i = cell_nodes[t];
    const double xi = cell_xy[t].x, yi = cell_xy[t].y;
    double R = 2.0 * h[i];
    double R2 = __dmul_rn(R, R);
    // float classification only where the float wrap cannot flip a candidate near the radius
    const bool filt = (!COPY || cell_xyf != nullptr) && (!g.periodic || R2 <= g.r2_wrap_max);
    const Prefilter pre((float)xi, (float)yi, (float)R2, g);
    int c = cell_of[i];
    int cx = c % g.nc[0], cy = c / g.nc[0];
    int xs[3], ys[3];
    int mx = axis_cells(cx, g.nc[0], g.periodic, xs);
    int my = axis_cells(cy, g.nc[1], g.periodic, ys);
    int cnt = 0;
    int64_t base = WRITE ? row_ptr[i] : 0;
    for (int a = 0; a < my; a++) {
        for (int b = 0; b < mx; b++) {
            int cc = ys[a] * g.nc[0] + xs[b];
            int64_t s = cell_start[cc], e = cell_start[cc + 1];
            for (int64_t p = s; p < e; p++) {
                int j = cell_nodes[p];
                if (j == i) continue;
                bool in;
                int decided = 0;  // 1: inside, 2: outside, 0: to the double test
                if (filt) {
                    bool inside, outside;
                    pre.test(float_at<COPY>(p, cell_xy, cell_xyf), g.periodic != 0, g, inside, outside);
                    decided = inside ? 1 : (outside ? 2 : 0);
                }
                if (decided) {
                    in = decided == 1;
                } else {
                    const double2 q = cell_xy[p];
                    in = within_exact(q.x, q.y, xi, yi, R2, g);
                }
                if (in) {
                    if (WRITE) col[base + cnt] = j;
                    cnt++;
                }
            }
        }
    }
    if (!WRITE) {
        counts[i] = cnt;
    } else {
        // insertion sort of the row (stencils hold tens of entries)
        int32_t *row = col + base;
        for (int u = 1; u < cnt; u++) {
            int32_t v = row[u];
            int w = u - 1;
            while (w >= 0 && row[w] > v) {
                row[w + 1] = row[w];
                w--;
            }
            row[w + 1] = v;
        }
    }
}

// Which of the two: whole searches take, with k_sweep_sparse and k_sweep, at 900^2 nodes 683 and 841 us at order 3 (6.8 nodes
// a cell), 762 and 893 at order 4 (7.8), but 1,057 and 932 at order 5 (10.2); at 600^2 order 2 and 3 (5.8, 6.8) 422 and 478,
// 443 and 470, at 450^2 364 and 335 at order 4; at 200^2 k_sweep wins at every order (194 against 259 at order 4).
// That mean counts empty cells too.  Rows of twice the pi nodes a node of the mean cell that a uniform set has at most (nnz, known
// to the write sweep, else 0) are those of a set that fills a part of its box, with many nodes in each cell: whole
// searches of 200,000 nodes, 100 to each of 5 % of the cells, took 3.4 ms with both sweeps by a thread per node, 0.8 with
// this one by k_sweep; 300 to each of 2 %, 28 and 4.3.
bool sparse_cells(int64_t n, const Grid &g, int64_t nnz)
{
    const double per_cell = (double)n / ((double)g.nc[0] * (double)g.nc[1]);
    if ((double)nnz > 2.0 * 3.15 * per_cell * (double)n) return false;
    return per_cell < 7.5 ? n >= 200000 : per_cell < 9.0 && n >= 400000;
}

unsigned sweep_blocks(int64_t n)
{
    const int64_t per = NB_THREADS / 32 * SWEEP_NODES;
    return (unsigned)((n + per - 1) / per);
}

template <bool WRITE, bool COPY>
void launch_sweep(int64_t n, const double *h, const Grid &g, const int32_t *cell_of, const int64_t *cell_start,
                  const int32_t *cell_nodes, const double2 *cell_xy, const float2 *cell_xyf, int32_t *counts,
                  const int64_t *row_ptr, int32_t *col, int64_t nnz, cudaStream_t s)
{
    if (sparse_cells(n, g, nnz))
        k_sweep_sparse<WRITE, COPY><<<(unsigned)((n + NB_THREADS - 1) / NB_THREADS), NB_THREADS, 0, s>>>(
            n, h, g, cell_of, cell_start, cell_nodes, cell_xy, cell_xyf, counts, row_ptr, col);
    else
        k_sweep<WRITE, COPY><<<sweep_blocks(n), NB_THREADS, 0, s>>>(n, h, g, cell_of, cell_start, cell_nodes, cell_xy, cell_xyf,
                                                              counts, row_ptr, col);
}

}  // namespace

// The float pre-filter's constants: E = 2^-21 (B + L) bounds |dx_float - dx| (B the largest
// coordinate magnitude of the box, L its larger side: the float roundings of both coordinates,
// of their difference and of the wrap, each at most 2^-24 of a magnitude below 2B + L), and the
// float test is used in a periodic box only for (2h)^2 <= (0.45 L_min)^2, where a candidate whose
// float and double wraps differ (|dx| within E of L/2) lies far outside the radius either way.
static void set_float_filter(Grid &g, const double lo[2], const double hi[2])
{
    double B = 0.0, Lmax = 0.0, Lmin = 1e300;
    for (int d = 0; d < 2; d++) {
        B = std::max(B, std::max(std::fabs(lo[d]), std::fabs(hi[d])));
        Lmax = std::max(Lmax, g.L[d]);
        Lmin = std::min(Lmin, g.L[d]);
        g.Lf[d] = (float)g.L[d];
        g.halfLf[d] = (float)g.halfL[d];
    }
    g.E = (float)std::ldexp(B + Lmax, -21);
    g.r2_wrap_max = (0.45 * Lmin) * (0.45 * Lmin);
}

labfm_status run_neighbours(labfm_ctx *ctx, int64_t n, const double *xy, const double *h, int periodic,
                            const double lo[2], const double hi[2], int64_t *nnz_out)
{
    cudaStream_t s = ctx->stream;
    ctx->n = 0;
    ctx->nnz = 0;
    LABFM_CUDA_TRY(ctx, ctx->misc.reserve(4096));
    unsigned long long *misc = ctx->misc.as<unsigned long long>();
    LABFM_CUDA_TRY(ctx, cudaMemsetAsync(misc, 0, 2 * sizeof(unsigned long long), s));
    int nb = (int)std::min<int64_t>((n + NB_THREADS - 1) / NB_THREADS, (int64_t)ctx->num_sms * 8);
    LABFM_CUDA_TRY(ctx, ctx->node_xy.reserve(sizeof(double2) * n));
    LABFM_CUDA_TRY(ctx, ctx->node_h.reserve(sizeof(double) * n));
    k_check<<<nb, NB_THREADS, 0, s>>>(n, xy, h, lo[0], lo[1], hi[0], hi[1], misc, ctx->node_xy.as<double2>(),
                                      ctx->node_h.as<double>());
    LABFM_CUDA_TRY(ctx, cudaGetLastError());
    unsigned long long *hs = (unsigned long long *)ctx->host_small;
    LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(hs, misc, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    if (hs[1] != 0)
        return fail(ctx, LABFM_ERR_ARG, std::to_string(hs[1]) + " node(s) with non-finite or out-of-box coordinates or h <= 0");
    double hmax;
    memcpy(&hmax, &hs[0], sizeof hmax);

    Grid g{};
    g.periodic = periodic;
    double ncell_d[2];
    for (int d = 0; d < 2; d++) {
        g.lo[d] = lo[d];
        g.L[d] = hi[d] - lo[d];
        g.halfL[d] = 0.5 * g.L[d];
        // side >= 2 h_max with a relative margin far above the rounding of the cell coordinate
        ncell_d[d] = std::floor(g.L[d] / (2.0 * hmax * (1.0 + 1e-9)));
        if (!(ncell_d[d] >= 1.0)) ncell_d[d] = 1.0;
    }
    // keep the grid to about 4 cells per node (coarser cells stay correct, just hold more nodes)
    double cap = 4.0 * (double)n + 64.0;
    if (ncell_d[0] * ncell_d[1] > cap) {
        double f = std::sqrt(ncell_d[0] * ncell_d[1] / cap);
        for (int d = 0; d < 2; d++) ncell_d[d] = std::max(1.0, std::floor(ncell_d[d] / f));
    }
    if (ncell_d[0] * ncell_d[1] > (double)(1 << 28))
        return fail(ctx, LABFM_ERR_CAPACITY, "cell grid exceeds 2^28 cells");
    for (int d = 0; d < 2; d++) {
        g.nc[d] = (int)ncell_d[d];
        g.inv_cs[d] = (double)g.nc[d] / g.L[d];
    }
    set_float_filter(g, lo, hi);
    int64_t ncells = (int64_t)g.nc[0] * g.nc[1];

    LABFM_CUDA_TRY(ctx, ctx->cell_of.reserve(sizeof(int32_t) * n));
    LABFM_CUDA_TRY(ctx, ctx->cell_count.reserve(sizeof(int32_t) * ncells));
    LABFM_CUDA_TRY(ctx, ctx->cell_start.reserve(sizeof(int64_t) * (ncells + 1)));
    LABFM_CUDA_TRY(ctx, ctx->cell_nodes.reserve(sizeof(int32_t) * n + sizeof(double2) * n + sizeof(float2) * n + 64));
    LABFM_CUDA_TRY(ctx, ctx->counts.reserve(sizeof(int32_t) * n));
    LABFM_CUDA_TRY(ctx, ctx->row_ptr.reserve(sizeof(int64_t) * (n + 2)));
    int32_t *cell_of = ctx->cell_of.as<int32_t>();
    int32_t *cell_count = ctx->cell_count.as<int32_t>();
    int64_t *cell_start = ctx->cell_start.as<int64_t>();
    int32_t *cell_nodes = ctx->cell_nodes.as<int32_t>();
    size_t xy_off = ((sizeof(int32_t) * n + 15) / 16) * 16;
    double2 *cell_xy = (double2 *)((char *)ctx->cell_nodes.ptr + xy_off);
    float2 *cell_xyf = (float2 *)(cell_xy + n);
    int32_t *counts = ctx->counts.as<int32_t>();
    int64_t *row_ptr = ctx->row_ptr.as<int64_t>();

    int nbn = (int)((n + NB_THREADS - 1) / NB_THREADS);
    LABFM_CUDA_TRY(ctx, cudaMemsetAsync(cell_count, 0, sizeof(int32_t) * ncells, s));
    // counts: the ranks until the sweep; behind the row offsets: the longest row
    k_cell_assign<<<nbn, NB_THREADS, 0, s>>>(n, xy, g, cell_of, cell_count, counts, row_ptr + n + 1);
    LABFM_CUDA_TRY(ctx, cudaGetLastError());
    LABFM_CUDA_TRY(ctx, exclusive_scan_i32_to_i64(cell_count, cell_start, ncells, ctx->scan_tmp, s));
    k_cell_scatter<<<nbn, NB_THREADS, 0, s>>>(n, xy, cell_of, cell_start, counts, cell_nodes, cell_xy, cell_xyf);
    LABFM_CUDA_TRY(ctx, cudaGetLastError());
    launch_sweep<false, true>(n, h, g, cell_of, cell_start, cell_nodes, cell_xy, cell_xyf, counts, nullptr, nullptr, 0, s);
    LABFM_CUDA_TRY(ctx, cudaGetLastError());
    LABFM_CUDA_TRY(ctx, exclusive_scan_i32_to_i64(counts, row_ptr, n, ctx->scan_tmp, s, reinterpret_cast<unsigned long long *>(row_ptr + n + 1)));
    int64_t *nnz_h = (int64_t *)ctx->host_small;
    LABFM_CUDA_TRY(ctx, cudaMemcpyAsync(nnz_h, row_ptr + n, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    const int64_t nnz = nnz_h[0];
    ctx->longest = nnz_h[1];
    if (nnz >= ((int64_t)1 << 40)) return fail(ctx, LABFM_ERR_CAPACITY, "too many stencil entries");
    LABFM_CUDA_TRY(ctx, ctx->col.reserve(sizeof(int32_t) * (nnz > 0 ? nnz : 1)));
    launch_sweep<true, true>(n, h, g, cell_of, cell_start, cell_nodes, cell_xy, cell_xyf, nullptr, row_ptr, ctx->col.as<int32_t>(), nnz, s);
    LABFM_CUDA_TRY(ctx, cudaGetLastError());
    LABFM_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    ctx->n = n;
    ctx->nnz = nnz;
    ctx->periodic = periodic;
    for (int d = 0; d < 2; d++) {
        ctx->lo[d] = lo[d];
        ctx->hi[d] = hi[d];
    }
    *nnz_out = nnz;
    return LABFM_OK;
}

}  // namespace labfm

// ---------------------------------------------------------------------------------------------
// labfm_build_neighbours_noalloc: the same kernels on a fixed scratch array instead of
// context-owned allocations.
// ---------------------------------------------------------------------------------------------
#include <mutex>

namespace {

constexpr int64_t NA_MAXN = LABFM_NOALLOC_MAX_NODES;
constexpr int64_t NA_MAXC = LABFM_NOALLOC_MAX_NODES;  // cells of the search grid
constexpr size_t na_align(size_t x) { return (x + 255) / 256 * 256; }
constexpr size_t NA_OFF_MISC = 0;
constexpr size_t NA_OFF_CELL_OF = na_align(NA_OFF_MISC + 64);
constexpr size_t NA_OFF_CELL_COUNT = na_align(NA_OFF_CELL_OF + 4 * NA_MAXN);
constexpr size_t NA_OFF_CELL_START = na_align(NA_OFF_CELL_COUNT + 4 * NA_MAXC);
constexpr size_t NA_OFF_CELL_NODES = na_align(NA_OFF_CELL_START + 8 * (NA_MAXC + 1));
constexpr size_t NA_OFF_CELL_XY = na_align(NA_OFF_CELL_NODES + 4 * NA_MAXN);
constexpr size_t NA_OFF_COUNTS = na_align(NA_OFF_CELL_XY + 16 * NA_MAXN);
constexpr size_t NA_OFF_SCAN = na_align(NA_OFF_COUNTS + 4 * NA_MAXN);
constexpr size_t NA_SCAN_ELEMS = 4096;
constexpr size_t NA_BYTES = na_align(NA_OFF_SCAN + 8 * NA_SCAN_ELEMS);  // about 10 MB

constexpr int NA_MAX_DEVICES = 64;
std::mutex g_na_mutex;  // serialises the address lookup (the array itself is not guarded)

struct DeviceGuard {
    int prev = -1;
    bool changed = false;
    ~DeviceGuard()
    {
        if (changed) cudaSetDevice(prev);
    }
};

}  // namespace

// The scratch of labfm_build_neighbours_noalloc (one copy per device that loads the library).
static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

extern "C" labfm_status labfm_build_neighbours_noalloc(int device, void *stream, int64_t n, const double *xy,
                                                       const double *h, int periodic, const double box_lo[2],
                                                       const double box_hi[2], int64_t *row_ptr, int32_t *col,
                                                       int64_t col_capacity, int64_t *nnz_out)
{
    using namespace labfm;
    if (n < 1 || !xy || !h || !box_lo || !box_hi || !row_ptr || !nnz_out || col_capacity < 0 ||
        (col_capacity > 0 && !col))
        return LABFM_ERR_ARG;
    if (n > NA_MAXN) return LABFM_ERR_CAPACITY;
    for (int d = 0; d < 2; d++)
        if (!std::isfinite(box_lo[d]) || !std::isfinite(box_hi[d]) || !(box_hi[d] > box_lo[d])) return LABFM_ERR_ARG;
    if (device < 0 || device >= NA_MAX_DEVICES) return LABFM_ERR_ARG;
    DeviceGuard guard;
    if (cudaGetDevice(&guard.prev) != cudaSuccess) return LABFM_ERR_CUDA;
    if (guard.prev != device) {
        if (cudaSetDevice(device) != cudaSuccess) return LABFM_ERR_CUDA;
        guard.changed = true;
    }
    // The array's device address, looked up on every call with the device current: in host code
    // g_noalloc_scratch names a host-side stand-in, and an address kept from an earlier call would
    // be stale after the device's primary context was reset (the module is then loaded again).
    // The first call on a device also loads the library's device code there.
    char *base;
    {
        std::lock_guard<std::mutex> lock(g_na_mutex);
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return LABFM_ERR_CUDA;
        base = static_cast<char *>(p);
    }
    cudaStream_t s = (cudaStream_t)stream;
    unsigned long long *misc = reinterpret_cast<unsigned long long *>(base + NA_OFF_MISC);
    int32_t *cell_of = reinterpret_cast<int32_t *>(base + NA_OFF_CELL_OF);
    int32_t *cell_count = reinterpret_cast<int32_t *>(base + NA_OFF_CELL_COUNT);
    int64_t *cell_start = reinterpret_cast<int64_t *>(base + NA_OFF_CELL_START);
    int32_t *cell_nodes = reinterpret_cast<int32_t *>(base + NA_OFF_CELL_NODES);
    double2 *cell_xy = reinterpret_cast<double2 *>(base + NA_OFF_CELL_XY);
    int32_t *counts = reinterpret_cast<int32_t *>(base + NA_OFF_COUNTS);
    int64_t *scan_tmp = reinterpret_cast<int64_t *>(base + NA_OFF_SCAN);

#define NA_TRY(expr)                                     \
    do {                                                 \
        if ((expr) != cudaSuccess) return LABFM_ERR_CUDA; \
    } while (0)

    int num_sms = 0;
    NA_TRY(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device));
    // node check and h_max (the counters start at zero on every call)
    NA_TRY(cudaMemsetAsync(misc, 0, 2 * sizeof(unsigned long long), s));
    int nb = (int)std::min<int64_t>((n + NB_THREADS - 1) / NB_THREADS, (int64_t)num_sms * 8);
    k_check<<<nb, NB_THREADS, 0, s>>>(n, xy, h, box_lo[0], box_lo[1], box_hi[0], box_hi[1], misc, nullptr, nullptr);
    NA_TRY(cudaGetLastError());
    unsigned long long hs[2];
    NA_TRY(cudaMemcpyAsync(hs, misc, sizeof hs, cudaMemcpyDeviceToHost, s));
    NA_TRY(cudaStreamSynchronize(s));
    if (hs[1] != 0) return LABFM_ERR_ARG;
    double hmax;
    memcpy(&hmax, &hs[0], sizeof hmax);

    // the same grid rule as labfm_build_neighbours, capped at the scratch's cell count
    Grid g{};
    g.periodic = periodic ? 1 : 0;
    double ncell_d[2];
    for (int d = 0; d < 2; d++) {
        g.lo[d] = box_lo[d];
        g.L[d] = box_hi[d] - box_lo[d];
        g.halfL[d] = 0.5 * g.L[d];
        ncell_d[d] = std::floor(g.L[d] / (2.0 * hmax * (1.0 + 1e-9)));
        if (!(ncell_d[d] >= 1.0)) ncell_d[d] = 1.0;
    }
    double cap = std::min(4.0 * (double)n + 64.0, (double)NA_MAXC);
    if (ncell_d[0] * ncell_d[1] > cap) {
        double f = std::sqrt(ncell_d[0] * ncell_d[1] / cap);
        for (int d = 0; d < 2; d++) ncell_d[d] = std::max(1.0, std::floor(ncell_d[d] / f));
    }
    for (int d = 0; d < 2; d++) {
        g.nc[d] = (int)ncell_d[d];
        g.inv_cs[d] = (double)g.nc[d] / g.L[d];
    }
    set_float_filter(g, box_lo, box_hi);
    const int64_t ncells = (int64_t)g.nc[0] * g.nc[1];
    if (ncells > NA_MAXC) return LABFM_ERR_CAPACITY;

    int nbn = (int)((n + NB_THREADS - 1) / NB_THREADS);
    NA_TRY(cudaMemsetAsync(cell_count, 0, sizeof(int32_t) * ncells, s));
    k_cell_assign<<<nbn, NB_THREADS, 0, s>>>(n, xy, g, cell_of, cell_count, counts, nullptr);  // counts: the ranks until the sweep
    NA_TRY(cudaGetLastError());
    NA_TRY(exclusive_scan_i32_to_i64_ws(cell_count, cell_start, ncells, scan_tmp, NA_SCAN_ELEMS, s));
    // (the float pre-filter's coordinates are converted where they are read: the fixed scratch holds no copy of them)
    k_cell_scatter<<<nbn, NB_THREADS, 0, s>>>(n, xy, cell_of, cell_start, counts, cell_nodes, cell_xy, nullptr);
    NA_TRY(cudaGetLastError());
    launch_sweep<false, false>(n, h, g, cell_of, cell_start, cell_nodes, cell_xy, nullptr, counts, nullptr, nullptr, 0, s);
    NA_TRY(cudaGetLastError());
    NA_TRY(exclusive_scan_i32_to_i64_ws(counts, row_ptr, n, scan_tmp, NA_SCAN_ELEMS, s));
    int64_t nnz = 0;
    NA_TRY(cudaMemcpyAsync(&nnz, row_ptr + n, sizeof nnz, cudaMemcpyDeviceToHost, s));
    NA_TRY(cudaStreamSynchronize(s));
    *nnz_out = nnz;
    if (nnz > col_capacity) return LABFM_ERR_CAPACITY;
    if (nnz > 0) {
        launch_sweep<true, false>(n, h, g, cell_of, cell_start, cell_nodes, cell_xy, nullptr, nullptr, row_ptr, col, nnz, s);
        NA_TRY(cudaGetLastError());
    }
    NA_TRY(cudaStreamSynchronize(s));
#undef NA_TRY
    return LABFM_OK;
}
