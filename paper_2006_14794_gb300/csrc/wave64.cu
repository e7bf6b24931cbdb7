// FP64 pairs of uniform lengths: the wavefront in registers, one cluster of
// thread blocks per pair (forward), one thread block per pair (backward).
//
// What bounds it.  A SM partition of this GPU takes 64 cycles for a warp's
// FP64 instruction (measured, dependent or not; four partitions together 19 a
// SM), so an FP64 sweep costs its number of FP64 operations, and moves,
// selects, shuffles and shared memory are free beside them.  Hence: few
// operations a cell, every lane at work in each of them, and at least one warp
// on each partition.
//
// Forms of the scheme.  Below dyadic order 2 the difference form (see
// fwd_chain.cu), three operations a cell,
//   sum = K(a,b-1) + K(a-1,b),  Q(a,b) = Q(a-1,b) + c sum,  K(a,b) = K(a,b-1) + Q(a,b);
// from order 2 on two,
//   K(a,b) = m K(a-1,b) + (m K(a,b-1) - K(a-1,b-1)),  m = 1 + c,
// where the rounding of 1 + c is carried along: what m lost of c is added to
// the coefficient of the row's next coarse cell before its own 1 + c (K varies
// little between them).  Against 80-bit arithmetic, 128-point paths, d = 8,
// order 2: 5.9e-14 relative for the scheme as printed, 1.3e-13 for m rounded
// plainly, 2.0e-14 with the carry, 5e-16 for the difference form.
//
// Schedule.  Warp g of a pair owns refined rows [32 R g, 32 R (g + 1)), lane l
// R consecutive ones; zero-increment rows are padded at the top.  At local
// step t lane l takes column t - l for all its rows, top to bottom, so a warp
// fills and drains in 31 steps whatever R is; the row above its first one
// comes by shuffle from lane l - 1, for lane 0 from the warp above through a
// ring in shared memory (at a block's edge in the neighbour block's, over the
// cluster).  Warps run W64_LAG steps behind one another with a barrier every
// W64_MAC: a value is written at least one barrier before it is read, and its
// ring slot is written again at least one barrier after.  Columns outside the
// grid have c = 0, which leaves K as it is, so lanes need no masks.
//
// Coefficients.  Every lane enters one new coarse column in each window of
// 2^lambda steps, at the step (lane mod 2^lambda) of it, and switches over by a
// select.  With many pairs (one warp each, several on a partition) all lanes
// form that column's R 2^-lambda coefficients together at the window's start,
// d DFMA each from shared memory: nothing is stored.  With few pairs that
// would leave the other partitions idle, so the whole block first forms the
// pair's coefficients in shared memory (PRE), and the rows can then be spread
// over more warps than coarse rows would fill.
//
// Measured (whole calls): a Gram of 64 x 64 paths of 128 points, d = 8, order 2:
// 63.6 ms with one block per pair and a barrier per anti-diagonal
// (fwd_plain.cu), 7.3 ms in the difference form with one warp a pair, 5.4 ms
// with m; its operations (2 a cell, d + 4 a coarse cell) take 4.9 ms.  8 x 8
// paths of 32 points, d = 3, order 1: 98 -> 31 us.  MMD^2 and its gradient, 16
// and 16 paths of 64 points, d = 32, order 1: 5.47 -> 1.03 ms (1.78 with the
// coefficients formed by the sweep warps alone).
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include "sigk_internal.cuh"

namespace cg = cooperative_groups;

namespace sigk {

namespace {

constexpr int W64_MAX_WARPS = 16;    // per block
constexpr int W64_MAX_CLUSTER = 8;   // blocks per pair (portable size)
constexpr int W64_MAC = 8;           // steps between barriers
constexpr int W64_LAG = 31 + 1 + W64_MAC;   // a multiple of W64_MAC, at least 31 + W64_MAC
constexpr int W64_RING = 64;         // columns kept between two warps
constexpr int W64_HELP = 256;        // least threads of a block that forms its coefficients first
constexpr int64_t W64_SMEM = 220 * 1024;
static_assert(W64_LAG % W64_MAC == 0 && W64_RING >= W64_LAG + W64_MAC, "ring slots live past their reader's barrier");

__host__ __device__ constexpr int w64_ng(int R, int lam) { return (R >> lam) > 0 ? R >> lam : 1; }   // coarse rows a lane
__host__ __device__ constexpr int w64_coarse(int R, int lam) { return (32 * R) >> lam; }              // a warp
__host__ __device__ constexpr bool w64_mform(int R, int lam) { return lam >= 2 && (R >> lam) > 0; }
// odd strides: staged columns one column apart, and rows one channel apart, hit distinct banks
__host__ __device__ inline int w64_odd(int64_t v) { return (int)(v | 1); }
__host__ __device__ inline int w64_nmac(int ny, int lam) { return ((ny << lam) + 31 + W64_MAC - 1) / W64_MAC; }
// Macro-steps before the first lane with a real row enters the grid: nothing to do,
// as the virtual rows above stay at K = 1 (less than 31 steps, so that a first warp
// without real rows still hands on all of its columns).
__host__ __device__ inline int w64_first(int vrows, int R, int lam) {
    const int m = (vrows << lam) / R / W64_MAC;
    return m < 3 ? m : 3;
}

// Shared memory of a block, in doubles: row increments (scaled) [d][coarse
// rows, odd], column increments [ny][d, odd], with the RBF lift the first
// points in the same layouts and the squared increments; the rings; the
// coefficients [ny][coarse rows, odd] where the block forms them first.
struct W64Shared { int64_t cols, pts, norms, ring, coef, total; int rs, ds; };
__host__ __device__ inline W64Shared w64_shared(int nrows, int warps, int ny, int64_t d, bool rbf, bool pre) {
    W64Shared s;
    s.rs = w64_odd(nrows);
    s.ds = w64_odd(d);
    s.cols = (int64_t)s.rs * d;
    s.pts = s.cols + (int64_t)ny * s.ds;
    s.norms = s.pts + (rbf ? s.pts : 0);
    s.ring = (s.norms + (rbf ? nrows + ny : 0) + 1) / 2 * 2;
    s.coef = s.ring + 2 * (int64_t)warps * W64_RING;
    s.total = s.coef + (pre ? (int64_t)ny * s.rs : 0);
    return s;
}

struct Wave64Args {
    PairSrc src;          // oriented: rows refine A, La <= Lb
    double *out;
    int64_t n_pairs;
    int nx, ny, vrows;    // coarse rows / columns, virtual coarse rows at the top
    int wpc, cluster;     // sweep warps per block, blocks per pair
    double scale, rbf_s;  // 1/2 4^-lambda, 1/(2 sigma^2)
};

// Padded coarse rows [P0, P0 + nrows) and all columns of a pair into shared
// memory: increments (the linear kernel's rows scaled, exactly), and with the
// RBF lift the points they start at and their squares.  A virtual row has a zero
// increment and with the lift the path's first point, so its coefficients are
// zero and what w64_coefs carries through it into the real rows of the same lane
// is theirs.  Ends with a barrier.
template <bool RBF>
__device__ __forceinline__ void w64_stage(double *sm, const W64Shared &L, const double *x, const double *y, int d,
                                          int nx, int ny, int vrows, int P0, int nrows, double scale) {
    const double f = RBF ? 1.0 : scale;
    for (int v = threadIdx.x; v < nrows * d; v += blockDim.x) {
        const int P = v / d, c = v - P * d, p = P0 + P - vrows;
        const bool in = p >= 0 && p < nx;
        const double *r = x + (int64_t)(in ? p : 0) * d + c;
        sm[c * L.rs + P] = in ? (r[d] - r[0]) * f : 0.0;
        if (RBF) sm[L.pts + c * L.rs + P] = r[0];   // a virtual row rests on the path's first point
    }
    for (int v = threadIdx.x; v < ny * d; v += blockDim.x) {
        const int q = v / d, c = v - q * d;
        const double *r = y + (int64_t)q * d + c;
        sm[L.cols + (int64_t)q * L.ds + c] = r[d] - r[0];
        if (RBF) sm[L.pts + L.cols + (int64_t)q * L.ds + c] = r[0];
    }
    __syncthreads();
    if (RBF) {
        for (int v = threadIdx.x; v < nrows + ny; v += blockDim.x) {
            const double *r = v < nrows ? sm + v : sm + L.cols + (int64_t)(v - nrows) * L.ds;
            const int st = v < nrows ? L.rs : 1;
            double s = 0.0;
            for (int c = 0; c < d; ++c) s = fma(r[c * st], r[c * st], s);
            sm[L.norms + v] = s;
        }
        __syncthreads();
    }
}

// |x| by its exponent bits (a NaN above all): an FP64 compare would cost an FP64
// instruction.
__device__ __forceinline__ int w64_size(double x) { return __double2hiint(x) & 0x7fffffff; }
constexpr int w64_pow2(int e) { return (1023 + e) << 20; }
// kappa at the end of a step less kappa at its start: exponents e0, e1 and their
// difference x (from a difference of 1 on, where little cancels, the two ends are
// exact to their own size).
__device__ __forceinline__ double w64_step(double e0, double e1, double x) {
    return w64_size(x) >= w64_pow2(0) ? exp(e1) - exp(e0) : exp(e0) * expm1(x);
}
// The second difference of kappa over the cell of points x, x + dx (channel
// stride rs) and y, y + dy as the difference of two steps, along the side whose
// kappa changes less from corner (p, q).  E = -s |x - y|^2 and A, B, C as in
// sigk_internal.cuh.  The product form kappa(p,q) (a b + (1 + a)(1 + b) e) is right
// where a, b and e are of order one; beside a jump of several bandwidths e^A e^B
// cancels against e^C (three corners near one another, the fourth five bandwidths
// off: 1e-9 relative, further off no digit is left) or overflows.  The corners'
// exponents are sums of these four, which leaves an error of their size times
// 2^-53; from a size (that of the row's earlier cells too) of 32 on, and where a
// corner's kappa counts or the sums are too large to tell, every exponent comes
// from its own distance. 
__device__ __noinline__ double w64_far_cell(const double *x, const double *dx, int rs, const double *y,
                                            const double *dy, int d, double rbf_s, double E, double A, double B,
                                            double C, int size) {
    const bool rows = fabs(A) >= fabs(B);   // steps along x, at y_q and at y_{q+1}; else along y
    double e0 = E, s0 = rows ? B : A, e1 = E + (rows ? A : B), s1 = s0 + C, f0 = e0 + s0, f1 = e1 + s1;
    if (size >= w64_pow2(5) && (fmax(fmax(e0, e1), fmax(f0, f1)) > -16.0 || size >= w64_pow2(20))) {
        e0 = e1 = f0 = f1 = 0.0;
        double w0 = 0.0, w1 = 0.0, ee = 0.0;
        for (int k = 0; k < d; ++k) {
            const double u = x[k * rs] - y[k], xv = dx[k * rs], yv = dy[k];
            const double e = rows ? xv : -yv, v = u + (rows ? -yv : xv);   // the step, and u at its other side
            const double a = u + e, b = v + e;
            e0 = fma(u, u, e0);
            e1 = fma(v, v, e1);
            f0 = fma(a, a, f0);
            f1 = fma(b, b, f1);
            w0 = fma(u, e, w0);
            w1 = fma(v, e, w1);
            ee = fma(e, e, ee);
        }
        e0 *= -rbf_s;
        e1 *= -rbf_s;
        f0 *= -rbf_s;
        f1 *= -rbf_s;
        s0 = -rbf_s * (2.0 * w0 + ee);
        s1 = -rbf_s * (2.0 * w1 + ee);
    }
    return w64_step(e1, f1, s1) - w64_step(e0, f0, s0);
}

// The coefficients of local coarse rows P .. P + N - 1 at column q (in the
// grid), the scheme's map applied.  With the RBF lift the second difference of
// kappa (rbf_second_difference), what consecutive rows share carried down:
// kappa(p+1, q) = kappa(p, q) (1 + b), expm1(A(p+1, q)) = a + e^A expm1(C).
// The product form and the carried values keep their digits while the exponents
// stay of order one: rows with |A| or |B| of 1 or more (a single cell: 2), or C's that
// could add up to it, are formed one by one (w64_far_cell), their exponents carried.
// Against 80-bit corners, 3 channels, points 0.1 to 10 bandwidths apart, steps of 0.01
// to 60: within 3e-13 of the value (of 0.001 for smaller ones), where the product form
// is off by anything.
template <int N, bool RBF>
__device__ __forceinline__ void w64_coefs(double (&c)[N], const double *sm, const W64Shared &L, int d, int nrows,
                                          int P, int q, double scale, double rbf_s, int scheme) {
    const double *dx = sm + P, *dy = sm + L.cols + (int64_t)q * L.ds;
    double g[N];
#pragma unroll
    for (int i = 0; i < N; ++i) g[i] = 0.0;
    if constexpr (!RBF) {
#pragma unroll 4
        for (int k = 0; k < d; ++k) {
            const double yv = dy[k];
#pragma unroll
            for (int i = 0; i < N; ++i) g[i] = fma(dx[k * L.rs + i], yv, g[i]);
        }
#pragma unroll
        for (int i = 0; i < N; ++i) c[i] = scheme_coef(g[i], scheme);
    } else {
        const double *x0 = sm + L.pts + P, *y0 = dy + L.pts;
        double uu = 0.0, uy = 0.0, ux[N];
#pragma unroll
        for (int i = 0; i < N; ++i) ux[i] = 0.0;
        for (int k = 0; k < d; ++k) {
            const double yv = y0[k], dv = dy[k];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const double u = x0[k * L.rs + i] - yv, xv = dx[k * L.rs + i];
                if (i == 0) {
                    uu = fma(u, u, uu);
                    uy = fma(u, dv, uy);
                }
                ux[i] = fma(u, xv, ux[i]);
                g[i] = fma(xv, dv, g[i]);
            }
        }
        constexpr int LOGN = N == 1 ? 0 : N == 2 ? 1 : N <= 4 ? 2 : N <= 8 ? 3 : 4;
        constexpr int FAR = N == 1 ? 1 : 0;   // 2^FAR: a single cell's 1 + a loses e^2, a carried one e a row
        static_assert(N <= 16, "LOGN");
        double A = rbf_s * (2.0 * uy - sm[L.norms + nrows + q]);
        bool far = w64_size(A) >= w64_pow2(FAR);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            ux[i] = -rbf_s * (2.0 * ux[i] + sm[L.norms + P + i]);   // B
            g[i] = 2.0 * rbf_s * g[i];                               // C
            far = far || w64_size(ux[i]) >= w64_pow2(FAR) || w64_size(g[i]) >= w64_pow2(FAR - LOGN);
        }
        if (far) {
            double E = -rbf_s * uu;
            int size = w64_size(E);
#pragma unroll
            for (int i = 0; i < N; ++i) {
                size = max(max(size, w64_size(A)), max(w64_size(ux[i]), w64_size(g[i])));
                c[i] = scheme_coef(w64_far_cell(x0 + i, dx + i, L.rs, y0, dy, d, rbf_s, E, A, ux[i], g[i], size) * scale,
                                   scheme);
                E += ux[i];
                A += g[i];
            }
            return;
        }
        double kap = exp(-rbf_s * uu), a = expm1(A);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const double b = expm1(ux[i]), e = expm1(g[i]);
            const double ea = (1.0 + a) * e;   // expm1(A + C) - expm1(A)
            c[i] = scheme_coef(kap * fma(a, b, (1.0 + b) * ea) * scale, scheme);
            kap = fma(kap, b, kap);
            a += ea;
        }
    }
}

// All coefficients of nrows padded coarse rows, the first `virt` of them virtual,
// into dst[q][P] (row stride ld): a warp takes 32 rows and four columns at a time,
// with the lift (whose cells cost several hundred FP64 operations) 32 real cells in
// the order of dst.
template <bool RBF>
__device__ __forceinline__ void w64_all_coefs(double *dst, int64_t ld, const double *sm, const W64Shared &L, int d,
                                              int nrows, int virt, int ny, double scale, double rbf_s, int scheme) {
    if constexpr (RBF) {
        const int real = nrows - virt;
        for (int v = threadIdx.x; v < virt * ny; v += blockDim.x) dst[v / virt * ld + v % virt] = 0.0;
        for (int v = threadIdx.x; v < real * ny; v += blockDim.x) {
            const int q = v / real, P = virt + v - q * real;
            double c[1];
            w64_coefs<1, true>(c, sm, L, d, nrows, P, q, scale, rbf_s, scheme);
            dst[q * ld + P] = c[0];
        }
    } else {
        constexpr int QB = 4;
        const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
        const int rb = (nrows + 31) / 32, qb = (ny + QB - 1) / QB;
        for (int u = threadIdx.x >> 5; u < rb * qb; u += nw) {
            const int r = u / qb, q0 = (u - r * qb) * QB;
            const int P = r * 32 + lane;
            const int Pc = P < nrows ? P : nrows - 1;
            const double *dx = sm + Pc;
            const double *dy[QB];
            double g[QB];
#pragma unroll
            for (int j = 0; j < QB; ++j) {
                dy[j] = sm + L.cols + (int64_t)(q0 + j < ny ? q0 + j : ny - 1) * L.ds;
                g[j] = 0.0;
            }
#pragma unroll 2
            for (int k = 0; k < d; ++k) {
                const double xv = dx[k * L.rs];
#pragma unroll
                for (int j = 0; j < QB; ++j) g[j] = fma(xv, dy[j][k], g[j]);
            }
#pragma unroll
            for (int j = 0; j < QB; ++j)
                if (P < nrows && q0 + j < ny) dst[(q0 + j) * ld + P] = scheme_coef(g[j], scheme);
        }
    }
}

// PRE: the block forms its coefficients in shared memory first (then R may be
// less than a coarse row's 2^lambda).
template <int R, int LAM, bool RBF, bool PRE>
__global__ void __launch_bounds__(W64_MAX_WARPS * 32) wave64_kernel(Wave64Args a) {
    constexpr int S = 1 << LAM, NG = w64_ng(R, LAM), PW = w64_coarse(R, LAM);
    constexpr bool MF = w64_mform(R, LAM);
    extern __shared__ __align__(16) double w64_sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int C = a.cluster;
    const int64_t k = blockIdx.x / C;
    const int rank = (int)(blockIdx.x - k * C);
    const int d = (int)a.src.d, ny = a.ny, nrows = a.wpc * PW;
    const int W = a.wpc * C, g = rank * a.wpc + warp;
    const W64Shared L = w64_shared(nrows, a.wpc, ny, d, RBF, PRE);
    double2 *ring = reinterpret_cast<double2 *>(w64_sm + L.ring);
    double *cf = w64_sm + L.coef;

    const PairRef pr = pair_ref<true>(a.src, k);
    w64_stage<RBF>(w64_sm, L, (const double *)a.src.A + pr.a_row0 * a.src.d,
                   (const double *)a.src.B + pr.b_row0 * a.src.d, d, a.nx, ny, a.vrows, rank * nrows, nrows, a.scale);
    if constexpr (PRE) {
        const int virt = a.vrows - rank * nrows;   // of the block's rows
        w64_all_coefs<RBF>(cf, L.rs, w64_sm, L, d, nrows, virt < 0 ? 0 : virt < nrows ? virt : nrows, ny, a.scale,
                           a.rbf_s, a.src.scheme);
    }
    auto barrier = [&]() {
        if (C > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    barrier();

    const bool mine = warp < a.wpc;   // a sweep warp (the others only helped with the coefficients)
    // where this warp's bottom row goes: the ring of warp g + 1
    double2 *down = nullptr;
    if (mine && g + 1 < W)
        down = warp + 1 < a.wpc ? ring + (warp + 1) * W64_RING : cg::this_cluster().map_shared_rank(ring, rank + 1);
    const double2 *up = ring + (mine ? warp : 0) * W64_RING;
    const int P = ((warp * 32 + lane) * R) >> LAM;   // the lane's first coarse row in the block

    double K[R], clo[NG], chi[NG], rest[NG], res = 1.0;
#pragma unroll
    for (int r = 0; r < R; ++r) K[r] = 1.0;
#pragma unroll
    for (int i = 0; i < NG; ++i) {
        chi[i] = MF ? 1.0 : 0.0;
        rest[i] = 0.0;
    }
    double kout = 1.0, qout = 0.0, kpre = 1.0;
    const int ol = lane & (S - 1), lq = lane >> LAM;
    const int nmac = w64_nmac(ny, LAM), total = nmac + W64_LAG / W64_MAC * (W - 1);
    const int tend = (ny << LAM) + 30;   // lane 31's step on the last column
    for (int m = w64_first(a.vrows, R, LAM); m < total; ++m) {
        const int mm = m - W64_LAG / W64_MAC * g;
        if (mine && mm >= 0 && mm < nmac) {
#pragma unroll 1
            for (int win = 0; win < W64_MAC / S; ++win) {
                const int t0 = mm * W64_MAC + win * S;
                const int q = (t0 >> LAM) - lq;
                const bool in = q >= 0 && q < ny;
                double c[NG];
                if constexpr (PRE) {
#pragma unroll
                    for (int i = 0; i < NG; ++i) c[i] = cf[(int64_t)(in ? q : 0) * L.rs + P + i];
                } else {
                    w64_coefs<NG, RBF>(c, w64_sm, L, d, nrows, P, in ? q : 0, a.scale, a.rbf_s, a.src.scheme);
                }
#pragma unroll
                for (int i = 0; i < NG; ++i) {
                    clo[i] = chi[i];
                    chi[i] = in ? c[i] : 0.0;
                    if constexpr (MF) {
                        const double full = chi[i] + rest[i];
                        chi[i] = 1.0 + full;
                        rest[i] = full - (chi[i] - 1.0);
                    }
                }
#pragma unroll
                for (int jj = 0; jj < S; ++jj) {
                    const int t = t0 + jj;
                    double kin = __shfl_up_sync(FULL, kout, 1), qin = 0.0;
                    if constexpr (!MF) qin = __shfl_up_sync(FULL, qout, 1);
                    double2 top = make_double2(1.0, 0.0);
                    if (g > 0) top = up[t & (W64_RING - 1)];
                    if (lane == 0) { kin = top.x; qin = top.y; }
                    const bool hi = jj >= ol;
                    if constexpr (MF) {
                        double diag = kpre;   // K(a-1, b-1)
                        kpre = kin;
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const double mc = hi ? chi[r / S] : clo[r / S];
                            const double v = fma(mc, K[r], -diag);
                            diag = K[r];
                            kin = fma(mc, kin, v);
                            K[r] = kin;
                        }
                    } else {
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const double cc = hi ? chi[r / S] : clo[r / S];
                            const double sum = K[r] + kin;
                            qin = fma(cc, sum, qin);
                            kin = K[r] + qin;
                            K[r] = kin;
                        }
                    }
                    kout = kin;
                    qout = qin;
                    if (t == tend) res = kout;
                    if (lane == 31 && down && t >= 31) down[(t - 31) & (W64_RING - 1)] = make_double2(kout, qout);
                }
            }
        }
        if (W > 1) barrier();
    }
    if (mine && g == W - 1 && lane == 31) {
        a.out[pr.out0] = res;
        if (pr.out1 >= 0) a.out[pr.out1] = res;
    }
}

// ---- the backward ----------------------------------------------------------
// One block per pair in flight, each with a slot of the workspace.  Four
// phases: the coefficients ([column][coarse row], all warps), the forward
// sweep in the difference form keeping every cell's sum K(a,b-1) + K(a-1,b)
// ([warp][step][row][lane]), the adjoint of the difference form (the strip
// adjoint of fwd_strip.cu) run through the same steps backwards, and the chain
// rule as two small contractions by all threads.  Keeping the sums (8 bytes a
// cell, written and read once in 256-byte rows) costs less than undoing the
// forward step, which would add three FP64 operations a cell to the adjoint's
// four.
struct Wave64BwdArgs {
    PairSrc src;             // oriented: rows refine A, La <= Lb
    const double *gout;
    double *dA, *dB;         // gradients of the row and column paths, or null
    double *ws;
    int64_t slot;            // doubles per block
    int64_t n_pairs;
    int nx, ny, vrows, W;    // W: sweep warps
    double scale, rbf_s;
};

struct W64Slot { int64_t coef, sums, gbar; };
__host__ __device__ inline W64Slot w64_slot(int R, int lam, int W, int nx, int ny, bool rbf) {
    W64Slot s;
    s.coef = (int64_t)ny * W * w64_coarse(R, lam);
    s.sums = (int64_t)W * W64_MAC * w64_nmac(ny, lam) * R * 32;
    s.gbar = (int64_t)nx * ny;
    const int64_t z = (int64_t)(nx + 1) * (ny + 1);   // the RBF chain rule's weights go where the sums were
    if (rbf && s.sums < z) s.sums = z;
    return s;
}

constexpr int W64B_MAX_WARPS = 8;

template <int R, int LAM, bool RBF>
__global__ void __launch_bounds__(W64B_MAX_WARPS * 32, 2) wave64_bwd_kernel(Wave64BwdArgs a) {
    constexpr int S = 1 << LAM, NG = w64_ng(R, LAM), PW = w64_coarse(R, LAM);
    constexpr int SHARE = R < S ? S / R : 1;   // lanes that share a coarse row
    extern __shared__ __align__(16) double w64_sm[];
    const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
    const int d = (int)a.src.d, nx = a.nx, ny = a.ny, W = a.W, nrows = W * PW;
    const W64Shared L = w64_shared(nrows, W, ny, d, RBF, false);
    double2 *ring = reinterpret_cast<double2 *>(w64_sm + L.ring);
    const W64Slot sl = w64_slot(R, LAM, W, nx, ny, RBF);
    double *Cm = a.ws + (int64_t)blockIdx.x * a.slot;
    double *Sm = Cm + sl.coef, *Gb = Sm + sl.sums;
    const int nmac = w64_nmac(ny, LAM), T = W64_MAC * nmac;
    const int total = nmac + W64_LAG / W64_MAC * (W - 1), m0 = w64_first(a.vrows, R, LAM);
    const int ol = lane & (S - 1), lq = lane >> LAM;
    const bool mine = g < W;
    const int P = ((g * 32 + lane) * R) >> LAM;
    const double *cw = Cm + (mine ? P : 0);
    double *sw = Sm + (int64_t)(mine ? g : 0) * T * R * 32 + lane;
    // the lane's coefficients of window w (zero outside the grid)
    auto window = [&](double (&c)[NG], int w) {
        const int q = w - lq;
        const bool in = mine && q >= 0 && q < ny;
#pragma unroll
        for (int i = 0; i < NG; ++i) c[i] = in ? cw[(int64_t)q * nrows + i] : 0.0;
    };

    for (int64_t k = blockIdx.x; k < a.n_pairs; k += gridDim.x) {
        const PairRef pr = pair_ref<true>(a.src, k);
        const double *x = (const double *)a.src.A + pr.a_row0 * a.src.d;
        const double *y = (const double *)a.src.B + pr.b_row0 * a.src.d;
        __syncthreads();   // the shared arrays and the slot are free again
        // 1. increments and coefficients
        w64_stage<RBF>(w64_sm, L, x, y, d, nx, ny, a.vrows, 0, nrows, a.scale);
        w64_all_coefs<RBF>(Cm, nrows, w64_sm, L, d, nrows, a.vrows, ny, a.scale, a.rbf_s, a.src.scheme);
        __syncthreads();
        // 2. forward, keeping the sums
        {
            double K[R], clo[NG], chi[NG], cnx[NG];
#pragma unroll
            for (int r = 0; r < R; ++r) K[r] = 1.0;
#pragma unroll
            for (int i = 0; i < NG; ++i) chi[i] = 0.0;
            window(cnx, g == 0 ? (m0 * W64_MAC) >> LAM : 0);   // the warp's first one
            double kout = 1.0, qout = 0.0;
            for (int m = m0; m < total; ++m) {
                const int mm = m - W64_LAG / W64_MAC * g;
                if (mine && mm >= 0 && mm < nmac) {
#pragma unroll 1
                    for (int win = 0; win < W64_MAC / S; ++win) {
                        const int t0 = mm * W64_MAC + win * S;
#pragma unroll
                        for (int i = 0; i < NG; ++i) {
                            clo[i] = chi[i];
                            chi[i] = cnx[i];
                        }
                        window(cnx, (t0 >> LAM) + 1);
#pragma unroll
                        for (int jj = 0; jj < S; ++jj) {
                            const int t = t0 + jj;
                            double kin = __shfl_up_sync(FULL, kout, 1), qin = __shfl_up_sync(FULL, qout, 1);
                            double2 top = make_double2(1.0, 0.0);
                            if (g > 0) top = ring[g * W64_RING + (t & (W64_RING - 1))];
                            if (lane == 0) { kin = top.x; qin = top.y; }
                            const bool hi = jj >= ol;
                            double *st = sw + (int64_t)t * R * 32;
#pragma unroll
                            for (int r = 0; r < R; ++r) {
                                const double c = hi ? chi[r / S] : clo[r / S];
                                const double sum = K[r] + kin;
                                st[r * 32] = sum;
                                qin = fma(c, sum, qin);
                                kin = K[r] + qin;
                                K[r] = kin;
                            }
                            kout = kin;
                            qout = qin;
                            if (lane == 31 && g + 1 < W && t >= 31)
                                ring[(g + 1) * W64_RING + ((t - 31) & (W64_RING - 1))] = make_double2(kout, qout);
                        }
                    }
                }
                if (W > 1) __syncthreads();
            }
        }
        __syncthreads();
        // 3. the adjoint: P(a,b) = c(a,b+1) A(a,b+1) + V(a+1,b), A(a,b) = A(a,b+1) + P(a,b),
        // V(a,b) = P(a,b) + c(a,b) A(a,b), dk/dc(a,b) += A(a,b) sum(a,b); V(Ni+1,Nj) = 1.
        // Columns after the grid have A = 0; those before it (c = 0) are not stored.
        {
            double A[R], clo[NG], chi[NG], cup[NG], cpre[NG], ahi[NG], alo[NG], sn[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                A[r] = 0.0;
                sn[r] = mine ? sw[((int64_t)(T - 1) * R + r) * 32] : 0.0;
            }
            // the coefficients that windows w + 1 (cup), w (chi) and w - 1 (clo) bring, w - 2's on the way
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                chi[i] = 0.0;
                ahi[i] = 0.0;
                alo[i] = 0.0;
            }
            window(clo, (T >> LAM) - 1);
            window(cpre, (T >> LAM) - 2);
            double vout = 0.0;
            const int Nj = ny << LAM;
            for (int m = 0; m < total - m0; ++m) {
                const int mm = nmac - 1 - (m - W64_LAG / W64_MAC * (W - 1 - g));
                if (mine && mm >= 0 && mm < nmac) {
#pragma unroll 1
                    for (int win = W64_MAC / S - 1; win >= 0; --win) {
                        const int t0 = mm * W64_MAC + win * S, w = t0 >> LAM;
#pragma unroll
                        for (int i = 0; i < NG; ++i) {
                            cup[i] = chi[i];
                            chi[i] = clo[i];
                            clo[i] = cpre[i];
                        }
                        window(cpre, w - 2);
#pragma unroll
                        for (int jj = S - 1; jj >= 0; --jj) {
                            const int t = t0 + jj;
                            double sm[R];
#pragma unroll
                            for (int r = 0; r < R; ++r) {
                                sm[r] = sn[r];
                                if (t > 0) sn[r] = sw[((int64_t)(t - 1) * R + r) * 32];
                            }
                            double v = __shfl_down_sync(FULL, vout, 1);
                            if (lane == 31) {
                                v = t - 31 == Nj - 1 ? 1.0 : 0.0;
                                if (g + 1 < W)
                                    v = t >= 31 ? ring[(g + 1) * W64_RING + ((t - 31) & (W64_RING - 1))].x : 0.0;
                            }
                            const bool hi = jj >= ol;
#pragma unroll
                            for (int r = R - 1; r >= 0; --r) {
                                const int i = r / S;
                                const double c = hi ? chi[i] : clo[i];
                                // the next column's: step jj + 1 of this window, or step 0 of the next
                                const double c1 = jj + 1 < S ? (jj + 1 >= ol ? chi[i] : clo[i])
                                                             : (ol == 0 ? cup[i] : chi[i]);
                                const double Pv = fma(c1, A[r], v);
                                A[r] += Pv;
                                v = fma(c, A[r], Pv);
                                const double acc = fma(A[r], sm[r], hi ? ahi[i] : alo[i]);
                                if (hi) ahi[i] = acc;
                                else alo[i] = acc;
                            }
                            vout = v;
                            if (lane == 0 && g > 0) ring[g * W64_RING + (t & (W64_RING - 1))].x = vout;
                        }
                        // coarse column w - lq is complete
                        const int q = w - lq;
                        double sum[NG];
#pragma unroll
                        for (int i = 0; i < NG; ++i) sum[i] = ahi[i];
#pragma unroll
                        for (int o = 1; o < SHARE; o *= 2) sum[0] += __shfl_xor_sync(FULL, sum[0], o);
                        if (q >= 0 && q < ny && lane % SHARE == 0) {
#pragma unroll
                            for (int i = 0; i < NG; ++i) {
                                const int p = P + i - a.vrows;
                                if (p >= 0) Gb[(int64_t)p * ny + q] = sum[i] * scheme_dcoef(chi[i], a.src.scheme);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < NG; ++i) { ahi[i] = alo[i]; alo[i] = 0.0; }
                    }
                }
                if (W > 1) __syncthreads();
            }
        }
        __syncthreads();
        // 4. the chain rule
        const double gk = a.gout[pr.out0];
        double *dx = a.dA ? a.dA + pr.a_row0 * a.src.d : nullptr;
        double *dy = a.dB ? a.dB + pr.b_row0 * a.src.d : nullptr;
        if constexpr (!RBF) {
            // four rows (columns) by one channel a thread; the staged rows hold the factor `scale`
            for (int side = 0; side < 2; ++side) {
                double *dst = side == 0 ? dx : dy;
                if (!dst) continue;
                const double f = side == 0 ? gk * a.scale : gk;
                const int n = side == 0 ? nx : ny, kn = side == 0 ? ny : nx;
                const int sr = side == 0 ? ny : 1, sk = side == 0 ? 1 : ny;   // Gb strides
                for (int v = tid; v < (n + 3) / 4 * d; v += blockDim.x) {
                    const int p0 = v / d * 4, c = v - v / d * d;
                    const double *e = side == 0 ? w64_sm + L.cols + c : w64_sm + c * L.rs + a.vrows;
                    const int se = side == 0 ? L.ds : 1;
                    const double *gp[4];
                    double s[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        gp[i] = Gb + (int64_t)(p0 + i < n ? p0 + i : n - 1) * sr;
                        s[i] = 0.0;
                    }
#pragma unroll 2
                    for (int kk = 0; kk < kn; ++kk) {
                        const double ev = e[kk * se];
#pragma unroll
                        for (int i = 0; i < 4; ++i) s[i] = fma(gp[i][(int64_t)kk * sk], ev, s[i]);
                    }
                    // dk/dx_i = dk/d dx_{i-1} - dk/d dx_i
                    double prev = 0.0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (p0 + i >= n) break;
                        atomicAdd(dst + (int64_t)(p0 + i) * d + c, f * (prev - s[i]));
                        prev = s[i];
                        if (p0 + i + 1 == n || i == 3) atomicAdd(dst + (int64_t)(p0 + i + 1) * d + c, f * s[i]);
                    }
                }
            }
        } else {
            // through kappa (see bwd_plain.cu): Z(i,j) = f W(i,j) kappa(x_i, y_j) / sigma^2
            // where the sums were, then dk/dx_i = sum_j Z(i,j) (y_j - x_i) and the mirror
            double *Z = Sm;
            const int la = nx + 1, lb = ny + 1;
            for (int v = tid; v < la * lb; v += blockDim.x) {
                const int i = v / lb, j = v - v / lb * lb;
                double w = 0.0, uu = 0.0;
                if (i >= 1 && j >= 1) w += Gb[(int64_t)(i - 1) * ny + j - 1];
                if (i < nx && j >= 1) w -= Gb[(int64_t)i * ny + j - 1];
                if (i >= 1 && j < ny) w -= Gb[(int64_t)(i - 1) * ny + j];
                if (i < nx && j < ny) w += Gb[(int64_t)i * ny + j];
                for (int c = 0; c < d; ++c) {
                    const double u = x[(int64_t)i * d + c] - y[(int64_t)j * d + c];
                    uu = fma(u, u, uu);
                }
                Z[v] = gk * a.scale * w * exp(-a.rbf_s * uu) * (2.0 * a.rbf_s);
            }
            __syncthreads();
            for (int side = 0; side < 2; ++side) {
                double *dst = side == 0 ? dx : dy;
                if (!dst) continue;
                const double *own = side == 0 ? x : y, *oth = side == 0 ? y : x;
                const int n = side == 0 ? la : lb, kn = side == 0 ? lb : la;
                const int sr = side == 0 ? lb : 1, sk = side == 0 ? 1 : lb;
                for (int v = tid; v < n * d; v += blockDim.x) {
                    const int i = v / d, c = v - v / d * d;
                    const double o = own[v];
                    const double *z = Z + (int64_t)i * sr;
                    double s = 0.0;
#pragma unroll 2
                    for (int kk = 0; kk < kn; ++kk) s = fma(z[(int64_t)kk * sk], oth[(int64_t)kk * d + c] - o, s);
                    atomicAdd(dst + v, s);
                }
            }
        }
    }
}

// (rows a lane R, dyadic order) instances: whole coarse rows for coefficients
// formed in the sweep, any power of two for coefficients formed first
#define SIGK_W64_INLINE(X) \
    X(1, 0) X(2, 0) X(4, 0) X(8, 0) X(16, 0) X(2, 1) X(4, 1) X(6, 1) X(8, 1) X(12, 1) X(16, 1) \
    X(4, 2) X(8, 2) X(12, 2) X(16, 2) X(8, 3) X(16, 3)
#define SIGK_W64_PRE(X) \
    X(1, 0) X(2, 0) X(4, 0) X(1, 1) X(2, 1) X(4, 1) X(1, 2) X(2, 2) X(4, 2) X(8, 2) X(2, 3) X(4, 3) X(8, 3)
#define SIGK_W64_BWD(X) \
    X(1, 0) X(2, 0) X(4, 0) X(8, 0) X(1, 1) X(2, 1) X(4, 1) X(8, 1) X(2, 2) X(4, 2) X(8, 2) X(2, 3) X(8, 3)

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        sms = 152;
    }
    return sms;
}

// Cycles of `ops` FP64 warp instructions of each of `warps` warps on a SM: 64.5
// each on a partition of its own, 19.2 a SM with every partition busy (both
// measured), and 60 a step for the shuffle and the rest.
double w64_cycles(double steps, double ops, double warps) {
    const double share = warps * (19.2 / 64.5);
    return steps * (64.5 * ops * (share > 1.0 ? share : 1.0) + 60.0);
}
// FP64 operations of one coarse cell's coefficient (RBF: four special functions)
double w64_coef_ops(double d, bool rbf) { return rbf ? 5.0 * d + 200.0 : d; }
// Cycles of the plain sweep (fwd_plain.cu) on the same pairs: two blocks a SM, a
// barrier per anti-diagonal, each refined cell with its coefficient anew (with the
// lift at order 0 a diagonal takes 665 operations' time at d = 63, 559 at d = 50).
double w64_plain_cycles(int64_t n, double nx, double ny, double d, int lam, bool rbf, int sms) {
    const double Ni = nx * (1 << lam), warps = Ni / 32 > 1 ? Ni / 32 : 1.0;
    const double on = n > sms ? 2.0 : 1.0, waves = ceil((double)n / (sms * on));
    const double share = warps * on * (19.2 / 64.5);
    return waves * (Ni + ny * (1 << lam)) * (64.5 * (rbf ? 9.0 * d + 100.0 : 3.0 * d + 10.0) * (share > 1.0 ? share : 1.0));
}

}  // namespace

// The cheapest of the instances and cluster shapes for these sizes by
// w64_cycles: one warp a pair where the pairs alone fill the partitions (least
// fill and drain), more warps, blocks and helpers a pair the fewer pairs there
// are.  False where the staged increments fit no block, and where they leave room
// for one or two warps a SM, which form their coefficients alone, and the plain sweep
// with its two pairs a SM is faster (195 pairs of 24 and 161 points, d = 63, order 0,
// with the lift: 5.6 ms against 4.1; 318 of 210 and 227, d = 51: 146 against 26; for
// 693 random shapes the default was then slower than plain by 15 % in one).
bool wave64_plan(int64_t n, int64_t La, int64_t Lb, int64_t d, int lam, int kernel, Wave64Plan &p) {
    if (La < 2 || Lb < 2 || lam < 0 || lam > 3 || La > Lb) return false;
    // longer paths are refused by the plain sweep, which would take them otherwise
    if (Lb > (1 << 20) || d > 4096 || 3 * 8 * (((La - 1) << lam) + 1) > 227 * 1024) return false;
    const bool rbf = kernel == SIGK_KERNEL_RBF;
    const int nx = (int)(La - 1), ny = (int)(Lb - 1);
    const int sms = sm_count();
    double best = 1e300, full = 0.0;   // (full: of lone warps, in whole waves)
    p.lam = lam;
    auto consider = [&](int R, bool pre) {
        const int pw = w64_coarse(R, lam), wt = (nx + pw - 1) / pw, ng = w64_ng(R, lam);
        const bool mf = w64_mform(R, lam);
        for (int C = 1; C <= W64_MAX_CLUSTER && n * C <= (1LL << 30); C *= 2) {
            const int wpc = (wt + C - 1) / C, W = wpc * C;
            if (wpc > W64_MAX_WARPS || (C > 1 && wt <= C / 2 * wpc)) continue;
            const int64_t bytes = 8 * w64_shared(wpc * pw, wpc, ny, d, rbf, pre).total;
            if (bytes > W64_SMEM) continue;
            const int threads = pre && wpc * 32 < W64_HELP ? W64_HELP : wpc * 32;
            int64_t bps = (228 * 1024) / (bytes + 1024);
            const int64_t regs = 65536 / (threads * (R > 8 || (rbf && !pre) ? 128 : 96));
            if (bps > regs) bps = regs;
            if (bps < 1) continue;
            const double load = (double)(n * C) / sms;             // blocks a SM has to run,
            const double on = load < 1 ? 1 : (load < bps ? load : (double)bps);   // at once,
            const double waves = load <= bps ? 1 : load / bps;     // and how often
            const double steps = (double)W64_MAC * (w64_nmac(ny, lam) - w64_first(W * pw - nx, R, lam)) +
                                 (double)W64_LAG * (W - 1);
            double ops = (mf ? 2.0 : 3.0) * R + (mf ? 4.0 * ng / (1 << lam) : 0.0), first = 0.0;
            if (pre) first = 19.2 * on * (double)(wpc * pw) * ny / 32 * (w64_coef_ops((double)d, rbf) + 1);
            else ops += ng * (rbf ? 3.0 * d + 140.0 : (double)d) / (1 << lam);
            const double cost = waves * (first + w64_cycles(steps, ops, on * wpc) + (C > 1 ? 30.0 : 6.0) * (W > 1) * steps);
            if (cost < best) {
                best = cost;
                full = !pre && bps * wpc <= 2 ? cost / waves * ceil(waves) : 0.0;
                if (rbf && ng == 1) full *= (5.0 * d + 135.0) / (3.0 * d + 140.0);
                p.R = R; p.pre = pre; p.wpc = wpc; p.cluster = C; p.threads = threads; p.smem = (int)bytes;
                p.vrows = W * pw - nx;
            }
        }
    };
#define X(r, l) if (l == lam) consider(r, false);
    SIGK_W64_INLINE(X)
#undef X
#define X(r, l) if (l == lam) consider(r, true);
    SIGK_W64_PRE(X)
#undef X
    return best < 1e300 && full <= 1.1 * w64_plain_cycles(n, nx, ny, (double)d, lam, rbf, sms);
}

cudaError_t launch_wave64(const PairSrc &src, const Wave64Plan &p, int64_t n, double *out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    Wave64Args a;
    a.src = src;
    a.out = out;
    a.n_pairs = n;
    a.nx = (int)(src.La - 1);
    a.ny = (int)(src.Lb - 1);
    a.vrows = p.vrows;
    a.wpc = p.wpc;
    a.cluster = p.cluster;
    a.scale = 0.5 / (double)(1 << (2 * p.lam));
    a.rbf_s = 0.5 / (src.sigma * src.sigma);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(n * p.cluster));
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = (size_t)p.smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)p.cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = p.cluster > 1 ? 1 : 0;
    auto go = [&](auto kern) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT);
        return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, kern, a);
    };
    const bool rbf = src.kernel == SIGK_KERNEL_RBF;
#define X(r, l)                                \
    if (!p.pre && p.R == r && p.lam == l)      \
        return rbf ? go(wave64_kernel<r, l, true, false>) : go(wave64_kernel<r, l, false, false>);
    SIGK_W64_INLINE(X)
#undef X
#define X(r, l)                                \
    if (p.pre && p.R == r && p.lam == l)       \
        return rbf ? go(wave64_kernel<r, l, true, true>) : go(wave64_kernel<r, l, false, true>);
    SIGK_W64_PRE(X)
#undef X
    return cudaErrorInvalidValue;
}

// The backward's schedule and workspace, by the same model.
bool wave64_bwd_plan(int64_t n, int64_t La, int64_t Lb, int64_t d, int lam, int kernel, Wave64BwdPlan &p) {
    if (La < 2 || Lb < 2 || lam < 0 || lam > 3 || n < 1) return false;
    if (La > Lb) { const int64_t t = La; La = Lb; Lb = t; }
    if (Lb > (1 << 15) || d > 4096) return false;
    const bool rbf = kernel == SIGK_KERNEL_RBF;
    const int nx = (int)(La - 1), ny = (int)(Lb - 1);
    const int sms = sm_count();
    double best = 1e300;
    p.lam = lam;
    // FP64 warp operations besides the sweeps, spread over all warps: coefficients and
    // chain rule
    const double cells = (double)nx * ny / 32, dd = (double)d;
    const double around = rbf ? cells * (w64_coef_ops(dd, true) + 6.0 * dd + 60.0) : cells * 3.0 * dd;
    auto consider = [&](int R, int threads) {
        const int pw = w64_coarse(R, lam), W = (nx + pw - 1) / pw;
        if (W * 32 > threads) return;
        const int64_t bytes = 8 * w64_shared(W * pw, W, ny, d, rbf, false).total;
        if (bytes > W64_SMEM) return;
        int64_t bps = (228 * 1024) / (bytes + 1024);
        if (bps > 65536 / (threads * 128)) bps = 65536 / (threads * 128);
        if (bps < 1) return;
        const W64Slot s = w64_slot(R, lam, W, nx, ny, rbf);
        const int64_t slot = (s.coef + s.sums + s.gbar + 31) / 32 * 32;
        int64_t grid = bps * sms;
        if (grid > n) grid = n;
        while (grid > 1 && grid * slot * 8 > W64_BWD_WS_CAP) grid = (grid + 1) / 2;
        if (grid * slot * 8 > 4 * W64_BWD_WS_CAP) return;
        const double on = (double)((grid + sms - 1) / sms), waves = (double)n / grid > 1 ? (double)n / grid : 1.0;
        const double steps = (double)W64_MAC * (w64_nmac(ny, lam) - w64_first(W * pw - nx, R, lam)) +
                             (double)W64_LAG * (W - 1);
        const double own = 64.5 * 32 / threads, shared = 19.2 * on;
        const double cost = waves * (around * (own > shared ? own : shared) + w64_cycles(steps, 3.0 * R, on * W) +
                                     w64_cycles(steps, 4.0 * R, on * W) + 12.0 * (W > 1) * steps);
        if (cost < best) {
            best = cost;
            p.R = R; p.W = W; p.threads = threads; p.smem = (int)bytes; p.slot = slot; p.grid = grid;
            p.vrows = W * pw - nx;
        }
    };
    // Fewer warps a block, and more blocks a SM, for pairs with less than two coarse cells a
    // thread of a full one (1310 pairs of 5 and 11 points, d = 9: 149 -> 62 us, 100 plain);
    // the slots of more blocks at once fall out of the L1 otherwise (801 pairs of 31 and
    // 242 points with the lift: 2.98 ms in full blocks, 3.49 in smaller ones).
    const int least = (int64_t)nx * ny <= 64 * W64B_MAX_WARPS ? 64 : 32 * W64B_MAX_WARPS;
#define X(r, l) if (l == lam) for (int t = 32 * W64B_MAX_WARPS; t >= least; t /= 2) consider(r, t);
    SIGK_W64_BWD(X)
#undef X
    return best < 1e300;
}

cudaError_t launch_wave64_bwd(const PairSrc &src, const Wave64BwdPlan &p, int64_t n, const double *gout, double *dA,
                              double *dB, void *ws, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    Wave64BwdArgs a;
    a.src = src;
    a.gout = gout;
    a.dA = dA;
    a.dB = dB;
    a.ws = (double *)ws;
    a.slot = p.slot;
    a.n_pairs = n;
    a.nx = (int)(src.La - 1);
    a.ny = (int)(src.Lb - 1);
    a.vrows = p.vrows;
    a.W = p.W;
    a.scale = 0.5 / (double)(1 << (2 * p.lam));
    a.rbf_s = 0.5 / (src.sigma * src.sigma);
    auto go = [&](auto kern) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT);
        if (e != cudaSuccess) return e;
        kern<<<(int)p.grid, p.threads, p.smem, st>>>(a);
        return cudaGetLastError();
    };
    const bool rbf = src.kernel == SIGK_KERNEL_RBF;
#define X(r, l)                  \
    if (p.R == r && p.lam == l)  \
        return rbf ? go(wave64_bwd_kernel<r, l, true>) : go(wave64_bwd_kernel<r, l, false>);
    SIGK_W64_BWD(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace sigk
