// FP64 weight build (Sec. 3.1-3.2), the device side: one node by a group of G threads.
//
// Per node: M = sum_j X_j (outer) W_j over its neighbours (Eq. disc_form), Gaussian elimination with
// partial pivoting of M Psi = C^d for all operators at once (Eq. lsys), and w_j^d = W_j . Psi^d (Eq. w_abf).
//
// A group of G threads per node (persistent over a node list): the whole CTA (G = 256) from order 6
// or 7 up, and two or four nodes per CTA below (G = 128 or 64, each group on its own named
// barrier), where the p x p system is small and a whole CTA would spend its time in barrier
// latency with most threads idle.  G per order is chosen by timing (build autotuner).
//
// Orders 1-3, and 4 with the full chain rule, form M from X and W themselves.  The others use two facts about the ABFs of Sec. 3.2:
//
// (1) The weights depend only on the space that the ABFs span: w_j = W_j . Psi with sum_j X_j w_j = C is
//     the same for every basis of that space.  The elements of degree n whose ABF is dW0/dr d^alpha|r|
//     are W0'(q) q^(1-2n) P_alpha(x, y) with the n + 1 independent homogeneous polynomials P_alpha of degree
//     n, so they span g_n x^a y^b, a + b = n, g_n = W0' q^(1-2n).  (With the full chain rule the elements of
//     degree 2 and 3 span four other radial functions times harmonics instead, see NLOWFAM.)
// (2) In that basis M_(a',b'),(a,b) = sum_j g_n x^(a+a') y^(b+b') = T_n(a + a', b + b'): its entries are moments,
//     and T_n(s, t) = T_(n+1)(s + 2, t) + T_(n+1)(s, t + 2), because g_n = g_(n+1) (x^2 + y^2).  So T_K at degrees
//     K + 1 .. 2K and the highest degree n + K of each other T_n are all the sums over neighbours there are:
//     199 at order 8 where M has 1936 entries; the rest are additions (no cancellation: x^2, y^2 >= 0).
//
// The weights are w_j = sum_n g_n sum_(a+b=n) Phi_ab x^a y^b = W0' r sum Phi_ab u^a v^b with (u, v) = (x, y) / r^2
// (g_n = g_1 r^(2-2n)), one polynomial in two variables by Horner's rule: neither X nor W of a neighbour is
// formed.  The FP64 pipe bounds the build (two lanes per SM and clock on GB300), and this takes its work at
// order 8 from 181 k to about 80 k multiply-adds per node.  The basis g_n x^a y^b is also better conditioned
// than the ABFs (median condition number at order 8, +-0.3 s noise: 1e10 against 3e12), so the weights come out
// closer to the exact ones (order 8: about ten times).  The orders below keep X and W: their systems are so small that
// nothing is gained, and the rounding of the recurrence shows there (5e-16 against 4e-16).
//
// Per-node orders (walls and variable resolution, Sec. 4.1) run in one persistent launch over
// work items: nodes bucketed by (order, stencil size), taken largest first, an item being one
// node of a CTA-wide order or 256 / G nodes of a grouped one.
#pragma once

#include <algorithm>

#include "abf.cuh"

namespace labfm {
struct BuildArgs {
    int64_t n_list;           // nodes in this launch
    const int32_t *list;      // node ids, or null: node = list index
    const double *xy;         // [2n]
    const double *h;          // [n]
    const int64_t *row_ptr;
    const int32_t *col;
    int periodic;
    double L[2], halfL[2];
    int rbf;
    int n_ops;
    void *w;  // [nnz][n_ops]
    int wdtype;
    int32_t *node_status;     // may be null
    unsigned long long *n_bad;
    double C[MAX_OPS * PMAX];  // target vectors, row d = C^d (physical units)
};

// Launchers of one form of the ABFs (the full chain rule in degrees 2 and 3, or every element
// dW0/dr d^alpha|r|), each form compiled in its own translation unit.  Orders 1-3 evaluate either form from
// BuildArgs::rbf: launch_order_dw0 serves both there.
struct OrderItems;
cudaError_t launch_order_dw0(int k, int G, const BuildArgs &a, int num_sms, cudaStream_t s);
cudaError_t launch_order_chain(int k, int G, const BuildArgs &a, int num_sms, cudaStream_t s);
cudaError_t launch_items_dw0(const BuildArgs &a, const OrderItems &I, int num_sms, cudaStream_t s);
cudaError_t launch_items_chain(const BuildArgs &a, const OrderItems &I, int num_sms, cudaStream_t s);
cudaError_t launch_any_dw0(const BuildArgs &a, const int8_t *order, int uniform_order, int num_sms, cudaStream_t s);
cudaError_t launch_any_chain(const BuildArgs &a, const int8_t *order, int uniform_order, int num_sms, cudaStream_t s);

// Work items of the one-launch build over per-node orders: orders from KMAX down; order k has
// n_items[k] items starting at item0[k], item t covering the list entries base[k] + (t -
// item0[k]) NG_k ... of that order, NG_k = 256 / group[k] (the last item may be short).
struct OrderItems {
    int group[KMAX + 1];
    int64_t base[KMAX + 1], cnt[KMAX + 1], item0[KMAX + 1], n_items[KMAX + 1];
    int64_t total;
};

constexpr int BUILD_THREADS = 256;
constexpr int FORM_MIN_ORDER = 4;  // from here on the kernels differ by the form of the ABFs (order 4 is built from moments in one of them)

// Orders built from moments: from 5 up, and order 4 where every ABF is dW0/dr d^alpha|r| (256^2 nodes: 1.55 ms against
// 2.08 from X and W; with the full chain rule, where half of the 14 elements are further functions, 2.29 against 2.13).
__host__ __device__ constexpr bool by_moments(int K, bool chain) { return K >= (chain ? 5 : 4); }

// group sizes a given order may run with
__host__ __device__ constexpr bool group_ok(int K, int G)
{
    return G == 256 || (G == 128 && K <= 6) || (G == 64 && K <= 4);
}

namespace {

// Small arrays of the node being built, in the group's share of the CTA's dynamic shared memory.
template <int P> struct NodeShared {
    double psi[P * MAX_OPS];     // Psi^d (Phi^d where built from moments)
    double low[7 * MAX_OPS];     // the coefficients of the chain-rule elements of degrees 2 and 3
    double invpiv[P];            // 1 / pivot of each column, reused by the back substitution
    double hpow[KMAX + 1];       // h^-n
    double inv;
    int flag;                    // bit 0: zero/non-finite pivot, bit 1: non-finite weight, bit 2: non-finite M
    unsigned char perm[2][P];    // the elimination's rows by position (two lists, alternating)
    unsigned ratios[BUILD_THREADS / 32];  // each warp's neighbours, see ratio_bit
};

// The CTA's dynamic shared memory (four CTAs fit an SM); a CTA of NG = 256 / G groups gives each group
// a 1/NG share.
constexpr size_t SMEM_CTA = 56 * 1024;

// The four further function families of the full chain rule's elements of degrees 2 and 3, by the harmonics
// they multiply (W', W'', W''' the radial derivatives of W0, r the scaled distance): degree 2 spans
// A2 (x^2 - y^2), A2 x y and B2 with A2 = (W'' - W'/r) / r^2 and B2 = W'' + W'/r (the Laplacian of W0); degree 3
// spans A3 (x^3 - 3 x y^2), A3 (3 x^2 y - y^3), B3 x and B3 y with A3 = (W''' - 3 W''/r + 3 W'/r^2) / r^3 and
// B3 = (W''' + W''/r - W'/r^2) / r.  Their moments with the rows X run over the degrees F + 1 .. F + K of the
// monomials for family F = 0 (B2), 1 (B3), 2 (A2), 3 (A3).  Only A2 (from degree 2 on) and A3 are summed over the
// neighbours: B2 = r^2 A2 + g_1 and B3 = r^2 A3 + 2 A2 (r in units of 2h), so the moments of the other two follow from
// those and T_1.
constexpr int NLOWFAM = 4;

// Sizes of the moment path at order K.
template <int K, bool CH> struct Mom {
    static constexpr int P = p_of_k(K);
    // items: one monomial x^s y^t of degree d = s + t per thread, degrees 2K down to K + 1 (T_K and the
    // highest degree of T_(d-K)); with the chain rule the further families' sums join them, see ChainItems
    static constexpr int NBASE = 3 * K * (K + 1) / 2;
    static constexpr int NSLOT = 2;  // sums of a chain-rule item
    // sums over the monomials of degree d, T's and the families'
    static __host__ __device__ constexpr int nsum(int d)
    {
        int c = (d > K) + (d > K && d < 2 * K);
        for (int f = 2; f < NLOWFAM; f++) c += d >= f + (f == 3) && d <= f + K;
        return c;
    }
    static __host__ __device__ constexpr int nitem()
    {
        if (!CH) return NBASE;
        int c = 0;
        for (int d = 1; d <= 2 * K; d++) c += (d + 1) * ((nsum(d) + NSLOT - 1) / NSLOT);
        return c;
    }
    static constexpr int NIT = nitem();
    static constexpr int SPAN = (NIT + 31) / 32 * 32;
    // staged row of a neighbour: x^0 .. x^2K, y^0 .. y^2K, g_1 .. g_K, A2, A3
    static constexpr int XO = 0, YO = 2 * K + 1, GO = 2 * YO, FO = GO + K;
    static constexpr int LD = (FO + (CH ? 2 : 0)) | 1;  // odd: consecutive neighbours on distinct banks
    // kept of a neighbour for the weights: u, v, W0' r, the seven chain-rule functions
    static constexpr int LP = CH ? 11 : 3;
    // T_n at degrees n + 1 .. n + K, n = 1 .. K, then the further families' moments
    static __host__ __device__ constexpr int cnt(int n) { return K * (n + 1) + K * (K + 1) / 2; }
    static __host__ __device__ constexpr int toff(int n)
    {
        return K * (n - 1) * (n + 2) / 2 + (n - 1) * K * (K + 1) / 2;
    }
    static __host__ __device__ constexpr int loff(int f)
    {
        return NT + K * f * (f + 1) / 2 + f * K * (K + 1) / 2;
    }
    static constexpr int NT = K * K * (K + 3) / 2 + K * K * (K + 1) / 2;
    // (behind the families' moments those of A2 at degree 2, which B3 needs)
    static constexpr int NLOW = CH ? NLOWFAM * K * (K + 1) / 2 + K * NLOWFAM * (NLOWFAM + 1) / 2 + 3 : 0;
    static constexpr int PSZ = 2 * NBASE + NLOW;  // the sums of one part
    // position of (degree d, power s of x) behind the first entry of T_n (n = F for a further family)
    static __host__ __device__ constexpr int at(int n, int d, int s)
    {
        return d * (d + 1) / 2 - (n + 1) * (n + 2) / 2 + s;
    }
    // first item of degree d
    static __host__ __device__ constexpr int istart(int d) { return (2 * K + 1) * (2 * K + 2) / 2 - (d + 1) * (d + 2) / 2; }
};
static_assert(Mom<8, false>::NBASE == 108 && Mom<8, false>::NT == 640 && Mom<8, false>::toff(9) == 640, "moment counts");
static_assert(Mom<8, true>::NLOW == 227 && Mom<4, true>::NIT == 63 && Mom<5, true>::NIT == 87, "moment counts");

// The chain rule's items: a monomial and up to NSLOT of the sums over it.  A warp's instruction takes the FP64 pipe's
// time for all 32 lanes whether or not a lane needs it, and the middle degrees have up to four sums where the
// others have one to three: in items of two sums all warps together take 6 FP64 instructions per neighbour at order 4, 9 at
// order 5 and 12 at order 6, where an item per monomial, with all four families summed, took 12, 14 and 15.
template <int K> struct ChainItems {
    using M = Mom<K, true>;
    static constexpr int NONE = 0xffff;
    struct Item {
        unsigned char s, t;              // powers of x and y (t = 255: no item)
        unsigned char fn[M::NSLOT];      // the functions' places in the staged row
        unsigned short to[M::NSLOT];     // the sums' places in a part, NONE: an unused slot
    };
    Item v[M::SPAN];
};
template <int K> constexpr ChainItems<K> make_chain_items()
{
    using M = Mom<K, true>;
    ChainItems<K> T{};
    for (int e = 0; e < M::SPAN; e++) {
        T.v[e].t = 255;
        for (int q = 0; q < M::NSLOT; q++) {
            T.v[e].fn[q] = M::GO;
            T.v[e].to[q] = ChainItems<K>::NONE;
        }
    }
    int e = 0;
    for (int d = 2 * K; d >= 1; d--)
        for (int s = 0; s <= d; s++) {
            int q = M::NSLOT;  // the current item's slots in use
            e--;
            auto put = [&](int fn, int to) {
                if (q == M::NSLOT) {
                    e++;
                    q = 0;
                    T.v[e].s = (unsigned char)s;
                    T.v[e].t = (unsigned char)(d - s);
                }
                T.v[e].fn[q] = (unsigned char)fn;
                T.v[e].to[q++] = (unsigned short)to;
            };
            if (d > K) put(M::GO + K - 1, M::istart(d) + s);
            if (d > K && d < 2 * K) put(M::GO + d - K - 1, M::NBASE + M::istart(d) + s);
            if (d == 2) put(M::FO, 2 * M::NBASE + M::NLOW - 3 + s);
            for (int f = 2; f < NLOWFAM; f++)
                if (d > f && d <= f + K) put(M::FO + f - 2, 2 * M::NBASE + M::loff(f) - M::NT + M::at(f, d, s));
            e++;
        }
    return T;
}
template <int K> __device__ const ChainItems<K> chain_items = make_chain_items<K>();

template <int K, int G, bool CH> struct Cfg {
    static constexpr int P = p_of_k(K);
    static constexpr int NG = BUILD_THREADS / G;  // nodes per CTA
    static_assert(G % 32 == 0 && BUILD_THREADS % G == 0, "groups of whole warps");
    static constexpr size_t GROUP_SMEM = (SMEM_CTA / NG) / 16 * 16;
    static constexpr int LDA = P + MAX_OPS + 1;  // augmented row stride
    static constexpr bool MOMENTS = by_moments(K, CH);
    using M = Mom<K, CH>;
    // the others: X and W of a neighbour, odd row stride (rows of consecutive neighbours on distinct banks);
    // one tile of 1 x TN elements of M per thread
    static constexpr int LDX = (P + 3) / 4 * 4 + 1;
    static constexpr int TN = K == 4 ? 7 : K == 3 ? 3 : 1;
    static constexpr int CG = (P + TN - 1) / TN;
    static_assert(MOMENTS || (P * CG <= 32 && CG * TN <= LDX), "one warp holds the tiles");
    // neighbours per staged chunk: what the group's share of the CTA's shared memory holds, <= 72
    static constexpr size_t FIXED = sizeof(NodeShared<P>) + (MOMENTS ? sizeof(double) * (M::NT + M::NLOW) : 0);
    static constexpr size_t PER_NB = sizeof(double) * (MOMENTS ? M::LD + M::LP : 2 * LDX);
    static constexpr int NB_FIT = (int)((GROUP_SMEM - FIXED) / PER_NB);
    static constexpr int NB = NB_FIT < 72 ? NB_FIT / 2 * 2 : 72;  // even
    static_assert(NB >= 24, "a chunk worth staging");
    // the augmented matrix reuses the staged rows (they are not read after the assembly)
    static_assert((size_t)P * LDA <= (size_t)NB * (MOMENTS ? M::LD : LDX), "augmented matrix fits the staging");
    // The sums run over the even and the odd neighbours of a chunk apart and are added at the end, whatever the
    // group size, so that the weights do not depend on it: by two sets of threads where the group holds
    // them, else by two accumulators of each thread.
    static constexpr int SETS = G / M::SPAN >= 2 ? 2 : 1;
    static constexpr int ACC = 2 / SETS;
    static_assert(!MOMENTS || M::SPAN <= G, "a thread per item");
    static_assert(!MOMENTS || (size_t)2 * M::PSZ <= (size_t)NB * M::LD, "partial sums fit the staging");
};

// Row scale of the moment form: a! b! / 2^n for element (a, b) of degree n (exact)
struct RowScale {
    double v[PMAX];
};
constexpr RowScale make_rowscale()
{
    const double f[KMAX + 1] = {1, 1, 2, 6, 24, 120, 720, 5040, 40320};
    RowScale T{};
    for (int e = 0; e < PMAX; e++) {
        const int n = elem_degree(e), a = elem_a(e);
        double s = f[a] * f[n - a];
        for (int t = 0; t < n; t++) s *= 0.5;
        T.v[e] = s;
    }
    return T;
}
__constant__ RowScale c_rowscale = make_rowscale();

// Finiteness from the exponent bits (integer instructions: on GB300 an FP64 compare occupies the
// scarce FP64 pipe as long as a multiply-add)
__device__ __forceinline__ bool finite_bits(double x)
{
    return ((unsigned long long)__double_as_longlong(x) & 0x7ff0000000000000ull) != 0x7ff0000000000000ull;
}

// 1 / a by Newton-Raphson iteration (r <- r + r (1 - a r), which squares the relative error of
// r at each step) from the single-precision reciprocal of a's leading 23 mantissa bits, formed
// with integer operations and the FP32 unit: two steps take the start's ~2^-22 to the rounding
// of the last step (within an ulp of 1/a) in four FP64 multiply-adds.  Used for the pivots, where
// one lane's division would hold the warp's share of the FP64 pipe for longer.  Subnormal a and
// |a| >= 2^1022 (a reciprocal at or below the normal range) take the division.
__device__ __forceinline__ double recip_newton(double a)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(a);
    const int ef = (int)((b >> 52) & 0x7ff);  // biased exponent of a
    if (ef < 1 || ef > 2044) return 1.0 / a;
    const float mf = __int_as_float(0x3f800000 | (int)((b >> 29) & 0x7fffff));  // 1.f of a, in [1, 2)
    const unsigned int rb = __float_as_uint(__frcp_rn(mf));                    // in (0.5, 1]
    // r0 = (1 / mf) 2^-(ef - 1023) with a's sign, assembled as a double
    const unsigned long long er = (unsigned long long)((int)((rb >> 23) & 0xff) - 127 - ef + 2046);
    double r = __longlong_as_double((long long)((b & 0x8000000000000000ull) | (er << 52) |
                                                ((unsigned long long)(rb & 0x7fffff) << 29)));
    double e = fma(-a, r, 1.0);
    r = fma(r, e, r);
    e = fma(-a, r, 1.0);
    return fma(r, e, r);
}

// Named barrier of group g of G threads: 1..2 for G = 128, 3..6 for G = 64 (an id is never used
// with two thread counts); the CTA-wide group uses the CTA barrier.
template <int G> __device__ __forceinline__ int group_bar(int g) { return (G == 128 ? 1 : 3) + g; }

// Barrier of one group: the CTA barrier for a CTA-wide group, named barrier `bar` of G threads
// otherwise.
template <int G> __device__ __forceinline__ void gsync(int bar)
{
    if constexpr (G == BUILD_THREADS) {
        __syncthreads();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(G) : "memory");
    }
}

// Offset of neighbour entry e from node i, minimum image in a periodic box.  |dx| > L/2 is tested on the bit
// patterns (non-negative doubles order like them): an FP64 compare takes the FP64 pipe's time.
__device__ __forceinline__ double min_image(double d, double L, double halfL)
{
    if ((__double_as_longlong(d) & 0x7fffffffffffffffll) > __double_as_longlong(halfL)) d -= copysign(L, d);
    return d;
}

__device__ __forceinline__ void offset_of(const BuildArgs &A, int64_t e, double xi, double yi, double &dx, double &dy)
{
    const int64_t j = A.col[e];
    dx = A.xy[2 * j] - xi;
    dy = A.xy[2 * j + 1] - yi;
    if (A.periodic) {
        dx = min_image(dx, A.L[0], A.halfL[0]);
        dy = min_image(dy, A.L[1], A.halfL[1]);
    }
}

// A set of neighbours with |y| = 2^e |x| for one e (on a diagonal, say) has rows of X that are equal up to a power of two:
// M is singular, and from X and W comes out so, its pivot exactly zero.  The products x^s y^t of the moments round
// apart, so such sets are told by their offsets: bit e + 15 for a ratio 2^e, two bits for any other.
__device__ __forceinline__ unsigned ratio_bit(double x, double y)
{
    const int r = (__double2hiint(x) & 0x7fffffff) - (__double2hiint(y) & 0x7fffffff), e = (r >> 20) + 15;
    return __double2loint(x) == __double2loint(y) && (r & 0xfffff) == 0 && (unsigned)e <= 30u ? 1u << e : 3u;
}

// One neighbour at offset (x, y) in units of 2h (so every monomial is at most 1): what the weights need of it
// into keep[], and with ROW its staged row for the moment sums.
template <int K, bool CH, bool ROW>
__device__ __forceinline__ void stage_neighbour(double x, double y, int rbf, double *__restrict__ row,
                                                double *__restrict__ keep)
{
    using M = Mom<K, CH>;
    const double r2 = fma(x, x, y * y);
    const double ir = rsqrt(r2);  // r2 = 0 (a neighbour on top of the node): inf, and every sum with it
    const double ir2 = ir * ir;
    double d1, d2, d3;
    rbf_derivs(rbf, 2.0 * (r2 * ir), d1, d2, d3);
    const double g1 = d1 * ir;
    keep[0] = x * ir2;
    keep[1] = y * ir2;
    keep[2] = g1 * r2;
    if constexpr (CH) {
        const double iq = 0.5 * ir;
        const double a2 = fma(-d1, iq, d2) * ir2, b2 = fma(d1, iq, d2);
        const double a3 = fma(3.0 * iq, fma(d1, iq, -d2), d3) * (ir2 * ir), b3 = fma(iq, fma(-d1, iq, d2), d3) * ir;
        const double xx = x * x, yy = y * y;
        keep[3] = a2 * (xx - yy);
        keep[4] = a2 * (x * y);
        keep[5] = b2;
        keep[6] = a3 * (x * fma(-3.0, yy, xx));
        keep[7] = a3 * (y * fma(3.0, xx, -yy));
        keep[8] = b3 * x;
        keep[9] = b3 * y;
        if constexpr (ROW) {
            row[M::FO] = a2;
            row[M::FO + 1] = a3;
        }
    }
    if constexpr (ROW) {
        double xp = 1.0, yp = 1.0, g = g1;
        row[M::XO] = row[M::YO] = 1.0;
#pragma unroll
        for (int s = 1; s <= 2 * K; s++) {
            xp *= x;
            yp *= y;
            row[M::XO + s] = xp;
            row[M::YO + s] = yp;
        }
#pragma unroll
        for (int n = 1; n <= K; n++) {
            row[M::GO + n - 1] = g;
            if (n < K) g *= ir2;
        }
    }
}

// The whole build of node i at order K by a group of G threads (group-local thread index `tid`,
// barrier `bar`): M and the targets into the augmented matrix, elimination, weights.  Ends synchronised
// (the group's shared memory is reused by its next node).
template <int K, int G, bool CH>
__device__ __forceinline__ void build_node(const BuildArgs &A, int64_t i, double *smem, int tid, int bar)
{
    using C = Cfg<K, G, CH>;
    using M = Mom<K, CH>;
    constexpr int P = C::P, NB = C::NB, LDA = C::LDA;
    double *Am = smem;  // [P][LDA]  augmented [M | Chat], over the staged rows
    // moments: rows [NB][LD], kept values [NB][LP], T; from X and W: Xs, Ws [NB][LDX]
    double *rows = smem;
    double *keep = rows + NB * M::LD;
    double *T = keep + NB * M::LP;
    double *Xs = smem, *Ws = Xs + NB * C::LDX;
    NodeShared<P> &sh =
        *reinterpret_cast<NodeShared<P> *>(C::MOMENTS ? T + M::NT + M::NLOW : Ws + NB * C::LDX);
    double *s_psi = sh.psi, *s_invpiv = sh.invpiv, *s_hpow = sh.hpow;
    int &s_flag = sh.flag;
    double &s_inv = sh.inv;

    const int n_ops = A.n_ops;
    const int W_ = P + n_ops;  // used columns of the augmented matrix
    {
        const int64_t rs = A.row_ptr[i], re = A.row_ptr[i + 1];
        const int ni = (int)(re - rs);
        if (ni < P) {
            for (int64_t t = tid; t < (int64_t)ni * n_ops; t += G) {
                if (A.wdtype == LABFM_F64) ((double *)A.w)[rs * n_ops + t] = 0.0;
                else ((float *)A.w)[rs * n_ops + t] = 0.0f;
            }
            if (tid == 0) {
                if (A.node_status) A.node_status[i] = LABFM_NODE_UNDERSAMPLED;
                atomicAdd(A.n_bad, 1ull);
            }
            return;
        }
        const double xi = A.xy[2 * i], yi = A.xy[2 * i + 1], hi = A.h[i];
        const double ihi = recip_newton(hi);
        if (tid == 0) {
            double s = 1.0;
            for (int t = 0; t <= K; t++) {
                s_hpow[t] = s;
                s *= ihi;
            }
            s_flag = 0;
        }
        const int nchunks = (ni + NB - 1) / NB;
        bool finite = true;  // of the entries of M this thread writes
        if constexpr (C::MOMENTS) {
            const double ihalf = 0.5 * ihi;
            // this thread's item: the monomial x^sx y^sy and the functions it is summed with (sy < 0: none)
            const int set = C::SETS > 1 ? tid / M::SPAN : 0;
            const int item = C::SETS > 1 ? tid - set * M::SPAN : tid;
            constexpr int NS = CH ? M::NSLOT : 2;
            int sx = item, sy = -1, fn[NS], to[NS];
            if (set < C::SETS && item < M::NIT) {
                if constexpr (CH) {
                    const auto it = chain_items<K>.v[item];
                    sx = it.s;
                    sy = it.t;
#pragma unroll
                    for (int q = 0; q < NS; q++) {
                        fn[q] = it.fn[q];
                        to[q] = it.to[q];
                    }
                } else {
                    int d = 2 * K;  // T_K, and up to degree 2K - 1 T_(d-K)
                    while (sx > d) sx -= d-- + 1;
                    sy = d - sx;
                    fn[0] = M::GO + K - 1;
                    to[0] = M::istart(d) + sx;
                    fn[1] = M::GO + (d < 2 * K ? d - K - 1 : 0);
                    to[1] = d < 2 * K ? M::NBASE + M::istart(d) + sx : ChainItems<K>::NONE;
                }
            }
            double acc[C::ACC][NS];
#pragma unroll
            for (int q = 0; q < C::ACC; q++)
#pragma unroll
                for (int f = 0; f < NS; f++) acc[q][f] = 0.0;
            unsigned ratios = 0;
            for (int ch = 0; ch < nchunks; ch++) {
                const int j0 = ch * NB, nj = min(NB, ni - j0);
                if (ch > 0) gsync<G>(bar);
                for (int t = tid; t < nj; t += G) {
                    double dx, dy;
                    offset_of(A, rs + j0 + t, xi, yi, dx, dy);
                    ratios |= ratio_bit(dx, dy);
                    stage_neighbour<K, CH, true>(dx * ihalf, dy * ihalf, A.rbf, rows + t * M::LD, keep + t * M::LP);
                }
                gsync<G>(bar);
                // one product and NS multiply-adds per item and neighbour
                if (sy >= 0) {
                    const double *rx = rows + M::XO + sx, *ry = rows + M::YO + sy;
                    const double *rf[NS];
#pragma unroll
                    for (int f = 0; f < NS; f++) rf[f] = rows + fn[f];
                    auto add = [&](int j, int q) {
                        const double m = rx[j * M::LD] * ry[j * M::LD];
#pragma unroll
                        for (int f = 0; f < NS; f++) acc[q][f] = fma(m, rf[f][j * M::LD], acc[q][f]);
                    };
                    // (NB is even, so a neighbour's parity is that of its place in the chunk)
                    if constexpr (C::SETS == 2) {
#pragma unroll 2
                        for (int j = set; j < nj; j += 2) add(j, 0);
                    } else {
                        int j = 0;
                        for (; j + 1 < nj; j += 2) {
                            add(j, 0);
                            add(j + 1, C::ACC - 1);
                        }
                        if (j < nj) add(j, 0);
                    }
                }
            }
            ratios = __reduce_or_sync(0xffffffffu, ratios);
            if ((tid & 31) == 0) sh.ratios[tid >> 5] = ratios;
            gsync<G>(bar);
            // the two parts' sums, over the staged rows
            if (sy >= 0) {
#pragma unroll
                for (int q = 0; q < C::ACC; q++) {
                    double *ps = rows + (C::SETS == 2 ? set : q) * M::PSZ;
#pragma unroll
                    for (int f = 0; f < NS; f++)
                        if (to[f] != ChainItems<K>::NONE) ps[to[f]] = acc[q][f];
                }
            }
            gsync<G>(bar);
            // The recurrence links T_n at degree d to T_(n-1) at degree d - 2: a warp follows each chain
            // c = d - 2n from its sum at the largest n down, a lane per power of x.
            {
                const int warp = tid >> 5, lane = tid & 31;
                for (int ci = warp; ci < 2 * K - 1; ci += G / 32) {
                    const int c = ci - (K - 1);
                    int n = c <= 0 ? K : K - c;
                    int dc = c + 2 * n;
                    const double *src = rows + (c <= 0 ? 0 : M::NBASE) + M::istart(dc) + lane;
                    double v = 0.0;
                    if (lane <= dc) {
                        v = src[0] + src[M::PSZ];
                        T[M::toff(n) + M::at(n, dc, lane)] = v;
                    }
                    while (n > 1 && dc - 2 >= n) {
                        v += __shfl_down_sync(0xffffffffu, v, 2);
                        n--;
                        dc -= 2;
                        if (lane <= dc) T[M::toff(n) + M::at(n, dc, lane)] = v;
                    }
                }
                if constexpr (CH)
                    for (int e = M::loff(2) - M::NT + tid; e < M::NLOW; e += G)
                        T[M::NT + e] = rows[2 * M::NBASE + e] + rows[M::PSZ + 2 * M::NBASE + e];
            }
            gsync<G>(bar);
            if constexpr (CH) {
                // B2 at degrees 1 .. K and B3 at degrees 2 .. K + 1 (T_1 at degree 1 from T_2)
                constexpr int NB2 = P, NB3 = P + K;
                for (int e = tid; e < NB2 + NB3; e += G) {
                    const bool b3 = e >= NB2;
                    int dd = b3 ? 2 : 1, ds = b3 ? e - NB2 : e;
                    while (ds > dd) ds -= dd++ + 1;
                    const double *up = T + (b3 ? M::loff(3) + M::at(3, dd + 2, ds) : M::loff(2) + M::at(2, dd + 2, ds));
                    double low;
                    if (b3) low = 2.0 * (dd == 2 ? T[M::NT + M::NLOW - 3 + ds] : T[M::loff(2) + M::at(2, dd, ds)]);
                    else if (dd == 1) low = T[M::toff(2) + M::at(2, 3, ds)] + T[M::toff(2) + M::at(2, 3, ds + 2)];
                    else low = T[M::toff(1) + M::at(1, dd, ds)];
                    T[b3 ? M::loff(1) + M::at(1, dd, ds) : M::loff(0) + M::at(0, dd, ds)] = (up[0] + up[2]) + low;
                }
                gsync<G>(bar);
            }
            // M from the moments: a warp per row (a', b'), a lane per column (a, b)
            {
                const int warp = tid >> 5, lane = tid & 31;
                constexpr int NQ = (P + 31) / 32;
                int cn[NQ], cb[NQ];  // degree of the column's element and its power of y
#pragma unroll
                for (int q = 0; q < NQ; q++) {
                    int n = 1, e = lane + 32 * q;
                    while (e > n) e -= n++ + 1;
                    cn[q] = n;
                    cb[q] = e;
                }
                int dm = 1, bm = warp;  // row m = warp: degree and power of y
                while (bm > dm) bm -= dm++ + 1;
                for (int m = warp; m < P; m += G / 32) {
                    const int am = dm - bm;
#pragma unroll
                    for (int q = 0; q < NQ; q++) {
                        const int c = lane + 32 * q, n = cn[q], b = cb[q];
                        if (c >= P) continue;
                        double v;
                        if (CH && (n == 2 || n == 3)) {
                            // the harmonics (x^2 - y^2, x y | 1) and (x^3 - 3 x y^2, 3 x^2 y - y^3 | x, y)
                            auto mom = [&](int f, int dd, int ds) {
                                return T[M::loff(f) + M::at(f, dm + dd, am + ds)];
                            };
                            if (n == 2)
                                v = b == 0   ? mom(2, 2, 2) - mom(2, 2, 0)
                                    : b == 1 ? mom(2, 2, 1)
                                             : mom(0, 0, 0);
                            else
                                v = b == 0   ? fma(-3.0, mom(3, 3, 1), mom(3, 3, 3))
                                    : b == 1 ? fma(3.0, mom(3, 3, 2), -mom(3, 3, 0))
                                             : mom(1, 1, b == 2 ? 1 : 0);
                        } else {
                            v = T[M::toff(n) + M::at(n, dm + n, am + n - b)];
                        }
                        Am[m * LDA + c] = v;
                        finite &= finite_bits(v);
                    }
                    bm += G / 32;
                    while (bm > dm) bm -= dm++ + 1;
                }
            }
            // targets: row (a, b) of X is x^a y^b / (a! b!) in units of h, here x^a y^b in units of 2h
            for (int t = tid; t < P * n_ops; t += G) {
                const int m = t / n_ops, d = t % n_ops;
                Am[m * LDA + P + d] = A.C[d * PMAX + m] * s_hpow[elem_degree(m)] * c_rowscale.v[m];
            }
        } else {
            // X and W of the chunk's neighbours into shared memory (thread per neighbour)
            auto stage = [&](int j0, int nj) {
                for (int t = tid; t < nj; t += G) {
                    double dx, dy;
                    offset_of(A, rs + j0 + t, xi, yi, dx, dy);
                    double *X = Xs + t * C::LDX, *W = Ws + t * C::LDX;
                    eval_xw<K>(dx * ihi, dy * ihi, A.rbf, X, W);
#pragma unroll
                    for (int e = P; e < C::LDX; e++) X[e] = W[e] = 0.0;
                }
            };
            const int rg = tid / C::CG, cg = tid % C::CG;
            const bool tile_active = tid < P * C::CG;
            double acc[C::TN];
#pragma unroll
            for (int b = 0; b < C::TN; b++) acc[b] = 0.0;
            for (int ch = 0; ch < nchunks; ch++) {
                const int j0 = ch * NB, nj = min(NB, ni - j0);
                if (ch > 0) gsync<G>(bar);
                stage(j0, nj);
                gsync<G>(bar);
                if (tile_active)
                    for (int j = 0; j < nj; j++) {
                        const double xv = Xs[j * C::LDX + rg];
                        const double *W = Ws + j * C::LDX + cg;
#pragma unroll
                        for (int b = 0; b < C::TN; b++) acc[b] = fma(xv, W[b * C::CG], acc[b]);
                    }
            }
            gsync<G>(bar);
            if (tile_active) {
#pragma unroll
                for (int b = 0; b < C::TN; b++) {
                    const int c = cg + b * C::CG;
                    if (c < P) {
                        Am[rg * LDA + c] = acc[b];
                        finite &= finite_bits(acc[b]);
                    }
                }
            }
            for (int t = tid; t < P * n_ops; t += G) {
                int m = t / n_ops, d = t % n_ops;
                Am[m * LDA + P + d] = A.C[d * PMAX + m] * s_hpow[elem_degree(m)];
            }
        }
        // a non-finite entry of M (a neighbour on top of node i: singular ABFs)
        if (!finite) atomicOr(&s_flag, 4);
        gsync<G>(bar);
        const bool bad_m = (s_flag & 4) != 0;

        // Gaussian elimination with partial pivoting (first largest |pivot| wins), the rows left in
        // place: a list of the rows by position (double-buffered, so that the update reads one list
        // while the next is written) stands for the exchanges.  The pivot search compares |entry|
        // as bit patterns (non-negative doubles order like their bits; a zero column gives 0, inf
        // and NaN sort above every finite value and are flagged): integer compares, where FP64
        // compares would take the FP64 pipe's time (7 % of the kernel at order 8, measured).
        // Look-ahead: in the step of column c the group's first warp updates column c + 1, finds
        // its pivot and scales it while the other warps update columns c + 2 on, so that a column
        // costs one group barrier.
        unsigned char *permA = sh.perm[0], *permB = sh.perm[1];
        // pivot of column c by the first warp: `pin` lists the rows by position, `pout` receives
        // the list with positions c and the pivot's exchanged; the column below the pivot is scaled
        auto pivot = [&](int c, const unsigned char *pin, unsigned char *pout) {
            unsigned long long best = 0ull;
            int bk = P;
            for (int k = c + tid; k < P; k += 32) {
                const unsigned long long v = (unsigned long long)__double_as_longlong(Am[pin[k] * LDA + c]) & 0x7fffffffffffffffull;
                if (v > best || (v == best && k < bk)) {
                    best = v;
                    bk = k;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
                if (ob > best || (ob == best && ok < bk)) {
                    best = ob;
                    bk = ok;
                }
            }
            if (bk >= P) bk = c;  // the same on every lane after the butterfly
            if (tid == 0) {
                if (best == 0ull || best >= 0x7ff0000000000000ull) {
                    s_flag |= 1;
                    s_inv = 0.0;
                } else {
                    s_inv = recip_newton(Am[pin[bk] * LDA + c]);
                }
                s_invpiv[c] = s_inv;
            }
            for (int k = tid; k < P; k += 32) pout[k] = pin[k == c ? bk : (k == bk ? c : k)];
            __syncwarp();
            const double inv = s_inv;
            for (int k = c + 1 + tid; k < P; k += 32) Am[pout[k] * LDA + c] *= inv;
        };
        if (!bad_m) {
            if (tid < 32) {
                for (int k = tid; k < P; k += 32) permB[k] = (unsigned char)k;
                __syncwarp();
                pivot(0, permB, permA);
            }
            gsync<G>(bar);
        }
        for (int c = 0; c + 1 < P && !bad_m; c++) {
            const unsigned char *cur = (c & 1) ? permB : permA;  // column c's pivot at position c
            unsigned char *nxt = (c & 1) ? permA : permB;
            const int pr = cur[c];
            const int nr = P - c - 1;
            if (tid < 32) {
                for (int k = c + 1 + tid; k < P; k += 32) {
                    const int r = cur[k];
                    Am[r * LDA + c + 1] = fma(-Am[r * LDA + c], Am[pr * LDA + c + 1], Am[r * LDA + c + 1]);
                }
                __syncwarp();
                pivot(c + 1, cur, nxt);
            } else {
                const int nc = W_ - c - 2;  // columns c + 2 .. W_ - 1
                for (int t = tid - 32; t < nr * nc; t += G - 32) {
                    const int k = c + 1 + t / nc, q = c + 2 + t % nc;
                    const int r = cur[k];
                    Am[r * LDA + q] = fma(-Am[r * LDA + c], Am[pr * LDA + q], Am[r * LDA + q]);
                }
            }
            gsync<G>(bar);
        }
        // back substitution on the n_ops right-hand sides, rows by final position: the column-c
        // step updates positions k < c with x_c; position c - 1 takes its last update there and is
        // scaled to x_(c-1) at once (the same product as scaling it at the start of the next step),
        // by the first n_ops threads apart from the others' updates: a multiply inside the shared
        // loop would take FP64 pipe time in every warp of the loop, masked or not
        const unsigned char *fp = ((P - 1) & 1) ? permB : permA;
        if (!bad_m) {
            if (tid < n_ops) Am[fp[P - 1] * LDA + P + tid] *= s_invpiv[P - 1];
            gsync<G>(bar);
        }
        for (int c = P - 1; c > 0 && !bad_m; c--) {
            const int rc = fp[c];
            if (tid < n_ops) {
                const int r = fp[c - 1];
                Am[r * LDA + P + tid] = fma(-Am[r * LDA + c], Am[rc * LDA + P + tid], Am[r * LDA + P + tid]) * s_invpiv[c - 1];
            }
            for (int t = tid; t < (c - 1) * n_ops; t += G) {
                const int k = t / n_ops, d = t % n_ops;
                const int r = fp[k];
                Am[r * LDA + P + d] = fma(-Am[r * LDA + c], Am[rc * LDA + P + d], Am[r * LDA + P + d]);
            }
            gsync<G>(bar);
        }
        bool one_ratio = false;
        if constexpr (C::MOMENTS) {
            unsigned ratios = 0;
#pragma unroll
            for (int w = 0; w < G / 32; w++) ratios |= sh.ratios[w];
            one_ratio = __popc(ratios) == 1;
        }
        const bool singular = (s_flag & 5) != 0 || one_ratio;  // no weights from a failed elimination
        for (int t = tid; t < P * n_ops; t += G) {
            const int m = t / n_ops, d = t - m * n_ops;
            double v = 0.0;  // a non-finite M gives no weights, and no position list is formed
            if (!bad_m) v = Am[fp[m] * LDA + P + d];
            if (C::MOMENTS && CH && m >= 2 && m < 9) {  // degrees 2 and 3: their own functions
                sh.low[(m - 2) * MAX_OPS + d] = v;
                v = 0.0;
            }
            s_psi[m * MAX_OPS + d] = v;
        }
        gsync<G>(bar);

        // weights: w_j^d = W0' r sum Phi_ab u^a v^b (+ the chain-rule functions), or W_j . Psi^d
        for (int ch = 0; ch < nchunks; ch++) {
            const int j0 = ch * NB;
            const int nj = min(NB, ni - j0);
            if (nchunks > 1) {  // what was kept of the other chunks' neighbours was overwritten: once more
                gsync<G>(bar);
                for (int t = tid; t < nj; t += G) {
                    double dx, dy;
                    offset_of(A, rs + j0 + t, xi, yi, dx, dy);
                    if constexpr (C::MOMENTS)
                        stage_neighbour<K, CH, false>(dx * (0.5 * ihi), dy * (0.5 * ihi), A.rbf, nullptr, keep + t * M::LP);
                    else
                        eval_xw<K>(dx * ihi, dy * ihi, A.rbf, Xs + t * C::LDX, Ws + t * C::LDX);
                }
                gsync<G>(bar);
            }
            for (int t = tid; t < nj * n_ops; t += G) {
                const int j = t / n_ops, d = t % n_ops;
                double s = 0.0;
                if (!singular) {
                    if constexpr (C::MOMENTS) {
                        const double *kp = keep + j * M::LP, *ph = s_psi + d;
                        const double u = kp[0], v = kp[1];
#pragma unroll
                        for (int b = K; b >= 0; b--) {  // Horner in u within Horner in v; no constant term
                            double r = ph[(p_of_k(K - 1) + b) * MAX_OPS];
#pragma unroll
                            for (int a = K - b - 1; a >= 0; a--) {
                                if (a + b > 0) r = fma(r, u, ph[(p_of_k(a + b - 1) + b) * MAX_OPS]);
                                else r *= u;
                            }
                            s = b == K ? r : fma(s, v, r);
                        }
                        s *= kp[2];
                        if constexpr (CH) {
#pragma unroll
                            for (int e = 0; e < 7; e++) s = fma(kp[3 + e], sh.low[e * MAX_OPS + d], s);
                        }
                    } else {
                        const double *W = Ws + j * C::LDX;
#pragma unroll
                        for (int m = 0; m < P; m++) s = fma(W[m], s_psi[m * MAX_OPS + d], s);
                    }
                    if (!finite_bits(s)) {
                        atomicOr(&s_flag, 2);
                        s = 0.0;
                    }
                }
                const int64_t idx = (rs + j0 + j) * n_ops + d;
                if (A.wdtype == LABFM_F64) ((double *)A.w)[idx] = s;
                else ((float *)A.w)[idx] = (float)s;
            }
        }
        gsync<G>(bar);
        const int flag = s_flag;
        if (flag & 2) {  // a weight was not finite: the whole node is zeroed
            for (int64_t t = tid; t < (int64_t)ni * n_ops; t += G) {
                if (A.wdtype == LABFM_F64) ((double *)A.w)[rs * n_ops + t] = 0.0;
                else ((float *)A.w)[rs * n_ops + t] = 0.0f;
            }
        }
        if (tid == 0) {
            int st = (flag & 4)   ? LABFM_NODE_NONFINITE
                     : (flag & 1) || one_ratio ? LABFM_NODE_SINGULAR
                     : (flag & 2) ? LABFM_NODE_NONFINITE
                                  : LABFM_NODE_OK;
            if (A.node_status) A.node_status[i] = st;
            if (st != LABFM_NODE_OK) atomicAdd(A.n_bad, 1ull);
        }
        gsync<G>(bar);  // shared state is reused by the next node
    }
}

// One order for all listed nodes (persistent over the list; 256 / G nodes per CTA at a time).
template <int K, int G, bool CH>
__global__ void __launch_bounds__(BUILD_THREADS, 4) k_build_fp64(BuildArgs A)
{
    using C = Cfg<K, G, CH>;
    extern __shared__ __align__(16) double smem[];
    const int g = threadIdx.x / G;
    double *gs = smem + g * (C::GROUP_SMEM / sizeof(double));
    for (int64_t li = (int64_t)blockIdx.x * C::NG + g; li < A.n_list; li += (int64_t)gridDim.x * C::NG)
        build_node<K, G, CH>(A, A.list ? (int64_t)A.list[li] : li, gs, threadIdx.x % G, group_bar<G>(g));
}

template <int K, int G, bool CH>
__device__ __forceinline__ void run_item(const BuildArgs &A, const OrderItems &I, int64_t t, double *smem)
{
    if constexpr (group_ok(K, G)) {
        using C = Cfg<K, G, CH>;
        const int g = threadIdx.x / G;
        const int64_t e = (t - I.item0[K]) * C::NG + g;  // entry within order K
        if (e < I.cnt[K])
            build_node<K, G, CH>(A, (int64_t)A.list[I.base[K] + e], smem + g * (C::GROUP_SMEM / sizeof(double)),
                             threadIdx.x % G, group_bar<G>(g));
    }
}

template <int K, bool CH>
__device__ __forceinline__ void run_item_k(const BuildArgs &A, const OrderItems &I, int64_t t, double *smem)
{
    switch (I.group[K]) {
    case 64: run_item<K, 64, CH>(A, I, t, smem); break;
    case 128: run_item<K, 128, CH>(A, I, t, smem); break;
    default: run_item<K, 256, CH>(A, I, t, smem); break;
    }
}

// Every order in one persistent launch: CTAs take the items in order (the costliest first, the
// list being bucketed by descending (order, stencil size)), so that the cheap ones fill the tail.
// The groups of a CTA run their items independently; where the group size changes from one item
// to the next, the whole CTA meets first, so that no group starts on shared memory (or a named
// barrier) that a group of the previous size still uses.  The item sequence, hence that barrier,
// is the same for every thread of the CTA.
template <bool CH>
__global__ void __launch_bounds__(BUILD_THREADS, 4) k_build_fp64_items(BuildArgs A, OrderItems I)
{
    extern __shared__ __align__(16) double smem[];
    int prev_group = 0;
    for (int64_t t = blockIdx.x; t < I.total; t += gridDim.x) {
        int k = KMAX;
        while (k > 1 && t >= I.item0[k] + I.n_items[k]) k--;
        if (I.group[k] != prev_group) {
            if (prev_group != 0) __syncthreads();
            prev_group = I.group[k];
        }
        switch (k) {
        case 1: run_item_k<1, false>(A, I, t, smem); break;
        case 2: run_item_k<2, false>(A, I, t, smem); break;
        case 3: run_item_k<3, false>(A, I, t, smem); break;
        case 4: run_item_k<4, CH>(A, I, t, smem); break;
        case 5: run_item_k<5, CH>(A, I, t, smem); break;
        case 6: run_item_k<6, CH>(A, I, t, smem); break;
        case 7: run_item_k<7, CH>(A, I, t, smem); break;
        default: run_item_k<8, CH>(A, I, t, smem); break;
        }
    }
}

// Listed nodes of any orders, one per CTA (the few nodes a mixed build hands back to FP64).
template <bool CH>
__global__ void __launch_bounds__(BUILD_THREADS, 4) k_build_fp64_any(BuildArgs A, const int8_t *__restrict__ order,
                                                                    int uniform_order)
{
    extern __shared__ __align__(16) double smem[];
    for (int64_t li = blockIdx.x; li < A.n_list; li += gridDim.x) {
        const int64_t i = A.list[li];
        switch (order ? order[i] : uniform_order) {
        case 1: build_node<1, 256, false>(A, i, smem, threadIdx.x, 0); break;
        case 2: build_node<2, 256, false>(A, i, smem, threadIdx.x, 0); break;
        case 3: build_node<3, 256, false>(A, i, smem, threadIdx.x, 0); break;
        case 4: build_node<4, 256, CH>(A, i, smem, threadIdx.x, 0); break;
        case 5: build_node<5, 256, CH>(A, i, smem, threadIdx.x, 0); break;
        case 6: build_node<6, 256, CH>(A, i, smem, threadIdx.x, 0); break;
        case 7: build_node<7, 256, CH>(A, i, smem, threadIdx.x, 0); break;
        default: build_node<8, 256, CH>(A, i, smem, threadIdx.x, 0); break;
        }
    }
}

template <class KernelT, class... Args>
cudaError_t launch_persistent_build(KernelT kern, int64_t units, int num_sms, cudaStream_t s, Args... args)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_CTA);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BUILD_THREADS, SMEM_CTA);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int64_t grid = std::min<int64_t>(units, (int64_t)num_sms * per_sm);
    if (grid < 1) return cudaSuccess;
    kern<<<(unsigned)grid, BUILD_THREADS, SMEM_CTA, s>>>(args...);
    return cudaGetLastError();
}

template <int K, bool CH>
cudaError_t launch_k(const BuildArgs &a, int G, int num_sms, cudaStream_t s)
{
    if (G == 64 && group_ok(K, 64))
        return launch_persistent_build(k_build_fp64<K, group_ok(K, 64) ? 64 : 256, CH>, (a.n_list + 3) / 4, num_sms, s, a);
    if (G == 128 && group_ok(K, 128))
        return launch_persistent_build(k_build_fp64<K, group_ok(K, 128) ? 128 : 256, CH>, (a.n_list + 1) / 2, num_sms, s,
                                       a);
    return launch_persistent_build(k_build_fp64<K, 256, CH>, a.n_list, num_sms, s, a);
}

template <bool CH>
cudaError_t launch_order(int k, int G, const BuildArgs &a, int num_sms, cudaStream_t s)
{
    switch (k) {
    case 1:
        if constexpr (!CH) return launch_k<1, false>(a, G, num_sms, s);
        return cudaErrorInvalidValue;
    case 2:
        if constexpr (!CH) return launch_k<2, false>(a, G, num_sms, s);
        return cudaErrorInvalidValue;
    case 3:
        if constexpr (!CH) return launch_k<3, false>(a, G, num_sms, s);
        return cudaErrorInvalidValue;
    case 4: return launch_k<4, CH>(a, G, num_sms, s);
    case 5: return launch_k<5, CH>(a, G, num_sms, s);
    case 6: return launch_k<6, CH>(a, G, num_sms, s);
    case 7: return launch_k<7, CH>(a, G, num_sms, s);
    default: return launch_k<8, CH>(a, G, num_sms, s);
    }
}

}  // namespace

}  // namespace labfm
