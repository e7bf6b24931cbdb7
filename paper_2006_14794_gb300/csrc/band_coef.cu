// The band form's coefficients (FP32): every coarse cell's c of every pair of
// a launch, written straight into the banded buffer that the sweeps of band.cu
// read (its layout: there), from the paths' points; linear kernel and RBF lift.
//
// A thread owns the slots of a lane l at one or more consecutive positions: the
// NG x NG cells (l NG + g, pos NG + w - g) of each, rows g and g + NG/2 as one
// float2 (FFMA2: the FP32 pipe's rate at half the issue slots, and the band's own
// order).  A warp covers 8 lanes by 4 positions (narrow lanes: 16 by 2): a read
// of the rows' float4s or of a position's column pairs is then one wavefront
// (32 lanes of one position took four for the rows), and a store meets 11 rows
// of the band where 32 lanes of one position would meet 32: those stores, not
// the FMAs, were what bounded the earlier form of this kernel.  Columns are kept
// as the pairs (column, column - NG/2) that rows g and g + NG/2 meet in a window.
// A block (one per SM at the larger sizes) walks a contiguous run of units, a
// unit being a pair's positions or, of long pairs, an even share of at most
// TILE of them.  Consecutive pairs of a Gram row share the row path and keep
// its staged values, and the next unit's column points arrive by cp.async
// while the current one is computed.
//
// RBF lift (Sec. 2.2; rbf_second_difference in sigk_internal.cuh): the second
// difference over cell (p, q) is kappa(p,q) (a b + (1 + a)(1 + b) e) with
//   a = expm1(A), A = s (2 <u,dy> - |dy|^2),   b = expm1(B), B = -s (2 <u,dx> + |dx|^2),
//   e = expm1(C), C = 2 s <dx,dy>,             u = x_p - y_q,
// and neighbouring cells share all but C: A(p+1,q) = A(p,q) + C(p,q), B(p,q+1)
// = B(p,q) + C(p,q), kappa(p,q+1) = kappa(p,q) (1 + a(p,q)), so
//   a(p+1,q) = a + (1 + a) e,   b(p,q+1) = b + (1 + b) e.
// Only a slot's first cell of each row takes kappa, a and b from the points,
// and its first row takes a in every column; every other cell adds its own
// <dx,dy> and about 14 operations.  Carried values keep FP32 accuracy while a
// and b stay of order one or below, so a slot with an |A| or |B| above KC_CARRY,
// or C's that could add up to it (data rough on the scale of the bandwidth),
// sums |u|^2 of every cell and forms each with its own exponentials, A and B
// moved on by C (kc_rough): 256 x 256 Gram of 128-point paths, d = 8, order 2, with a
// bandwidth of 0.2 where the paths span 1: 9.3 ms, 38 with such cells one at a
// time from their points, 10.8 before cells were carried at all, when each formed
// all six sums (9 d operations), three series and two exponentials and stored its
// value alone into a zero-filled band.
//
// Measured: the lift over 3840 pairs of 256-point paths, d = 32, order 1, 2.9 ->
// 1.16 ms; over a 256 x 256 Gram of 128-point paths, d = 8, order 2, 7.4 (zero
// fill included) -> 2.9 ms; the linear kernel over the 3840 pairs 0.62 -> 0.54 ms
// (0.67 in this form with 32 lanes of one position a warp).
// Padding: rows and columns outside the path repeat its end points, so their
// increments and with them c are exactly zero.
#include "rbf.cuh"
#include "sigk_internal.cuh"

namespace sigk {

namespace {

constexpr int KC_CH = 32;          // channels staged at a time by the linear kernel (the lift: all)
// Lanes a warp covers, positions a thread, most positions a unit, most warps a
// block.  12 warps a SM have 168 registers each; a pair of 33 positions (256
// points at dyadic order 1) is 36 warp items, three a warp.  Narrow lanes run 18
// warps a SM: two blocks of 9, or with the lift's shared memory one of 18.
template <int NG, bool RBF>
struct KcShape {
    static constexpr int LW = NG == 8 ? 8 : 16, NP = NG == 8 ? 1 : NG == 4 ? 2 : 4;
    static constexpr int GP = 32 / LW * NP;   // positions a warp item
    static constexpr int TILE = 36, TILEC = 12;   // (TILEC: with more channels than are staged at once)
    static constexpr int WARPS = NG == 8 ? 12 : RBF ? 18 : 9, MINB = NG == 8 || RBF ? 1 : 2;
};
constexpr float KC_CARRY = 0.5f;   // see above: a, b <= e^1 - 1 along a slot

struct KcArgs {
    PairSrc src;
    float *band;
    int64_t n_pairs;
    int TperR, NQV, vrows;
    int tiles, tp, passes;   // units a pair, positions a unit, items a warp
    int chunks, xch;         // channel chunks of a unit (more than one: one pass); row channels kept
    float scale, s;       // 1/2 4^-lambda, 1/(2 sigma^2)
};

__device__ __forceinline__ void kc_cp4(float *dst, const float *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void kc_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void kc_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <int NG>
__host__ __device__ constexpr int kc_xs() { return 32 * NG + 4; }
// a unit's columns, from NG - 1 before its first position's, and one more for
// the last increment (tp: rounded up to whole threads' positions)
__host__ __device__ inline int kc_ys(int tp, int NG) { return (tp * NG + NG + 3) / 4 * 4 + 4; }
// per channel: rows' increments, the next unit's column points, pairs of column
// increments; lift: and this unit's column points (as pairs too where they
// fit: not for NG = 8), row points, the squares
template <int NG>
__host__ __device__ constexpr int kc_pp() { return NG == 8 ? 1 : 2; }
template <int NG, bool RBF>
__host__ __device__ inline int kc_smem_floats(int tp, int nch, int xch) {
    const int ys = kc_ys(tp, NG), xs = kc_xs<NG>();
    return RBF ? nch * (3 + kc_pp<NG>()) * ys + 2 * xch * xs + ys + xs : nch * 3 * ys + xch * xs;
}
// threads that share a staged point's channels: the power of two at or above nc (32 at most)
__device__ __forceinline__ int kc_group(int nc) { return nc > 16 ? 32 : nc > 8 ? 16 : nc > 4 ? 8 : 4; }

// Where padded row P is staged: a lane's rows in the band's order (g, g + NG/2
// side by side), and with 8 of them the two 16-byte halves swapped for lanes
// 4..7 of every 8, so that the 8 lanes of a phase read 8 distinct bank quads.
template <int NG>
__device__ __forceinline__ int kc_xpos(int P) {
    const int l = P / NG, g = P - l * NG;
    const int at = g < NG / 2 ? 2 * g : 2 * (g - NG / 2) + 1;
    return l * NG + (NG == 8 ? at ^ (l & 4) : at);
}
// the lane's rows as pairs (h, h + NG/2)
template <int NG>
__device__ __forceinline__ void kc_rows(float2 (&v)[NG / 2], const float *r, int l) {
    if constexpr (NG >= 4) {
        const int sw = NG == 8 ? (l >> 2) & 1 : 0;
#pragma unroll
        for (int h = 0; h < NG / 4; ++h) {
            const float4 t = *reinterpret_cast<const float4 *>(r + l * NG + 4 * (h ^ sw));
            v[2 * h] = make_float2(t.x, t.y);
            v[2 * h + 1] = make_float2(t.z, t.w);
        }
    } else {
        v[0] = *reinterpret_cast<const float2 *>(r + l * NG);
    }
}
// N column pairs from r (16-byte aligned for NG > 2)
template <int NG, int N>
__device__ __forceinline__ void kc_cols(float2 (&v)[N], const float2 *r) {
    if constexpr (NG == 2) {
#pragma unroll
        for (int h = 0; h < N; ++h) v[h] = r[h];
        return;
    }
#pragma unroll
    for (int h = 0; h < N / 2; ++h) {
        const float4 t = *reinterpret_cast<const float4 *>(r + 2 * h);
        v[2 * h] = make_float2(t.x, t.y);
        v[2 * h + 1] = make_float2(t.z, t.w);
    }
    if constexpr (N % 2) v[N - 1] = r[N - 1];
}

__device__ __forceinline__ float2 kc2(float v) { return make_float2(v, v); }
// e^x - 1 of two values, |x| <= KC_CARRY / 2^(8 - D) or so: the Taylor series
// through x^D / D!, whose truncation is x^D / (D + 1)! of the value: 1.1e-8 for
// D = 8 and |x| <= 1/2 (a fifth of a rounding), below 2e-9 for D = 7 and 1/4, D = 6
// and 1/8, D = 5 and 1/16.
template <int D>
__device__ __forceinline__ float2 kc_expm1(float2 x) {
    constexpr float F[9] = {1.f, 1.f, 1.f / 2.f, 1.f / 6.f, 1.f / 24.f, 1.f / 120.f, 1.f / 720.f, 1.f / 5040.f,
                            1.f / 40320.f};
    float2 p = kc2(F[D]);
#pragma unroll
    for (int i = D - 1; i >= 1; --i) p = __ffma2_rn(p, x, kc2(F[i]));
    return __fmul2_rn(p, x);
}

// A slot's values v[w][h] = (cell (w, h), cell (w, h + NG/2)) to the band: its
// own slot; position 0 leaves the cells w < g to the previous pair (pair 0:
// zeros); position TperR is the pair's tail (w < g), in slot 0 of the next
// pair (after the last pair the slot has no owner and its other cells are
// zeroed).  Virtual columns (in positions 0 and 1) are zero whatever the points: the
// adjoint multiplies the first one with the previous pair's zero A, and a NaN or an
// infinity must stay in the pair whose path holds it.
template <int NG>
__device__ __forceinline__ void kc_store(float *band, int64_t k, int64_t n_pairs, int TperR, int NQV, int pos, int l,
                                         const float2 (&v)[NG][NG / 2]) {
    constexpr int SLOT = NG * NG, NH = NG / 2;
    float *dst = band + band_row(k * TperR + pos, l, NG, n_pairs * TperR + 1);   // (the tail: the next pair's slot 0)
    if (pos > (NQV > 1) && pos < TperR) {
#pragma unroll
        for (int i = 0; i < SLOT / 4; ++i) {
            const float2 u = v[2 * i / NH][2 * i % NH], t = v[(2 * i + 1) / NH][(2 * i + 1) % NH];
            *reinterpret_cast<float4 *>(dst + band_off(4 * i)) = make_float4(u.x, u.y, t.x, t.y);
        }
        return;
    }
    const bool tail = pos == TperR;
    const bool zero = tail ? k == n_pairs - 1 : k == 0;
#pragma unroll
    for (int w = 0; w < NG; ++w)
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const float c = g < NH ? v[w][g % NH].x : v[w][g % NH].y;
            const int at = band_off(w * NG + 2 * (g % NH) + g / NH);
            if (tail ? w < g : pos > 0 || w >= g) dst[at] = pos * NG + w - g < NQV ? 0.f : c;
            else if (zero) dst[at] = 0.f;
        }
}

// The scheme's map, then to the band.
template <int NG>
__device__ __forceinline__ void kc_put(const KcArgs &a, float2 (&v)[NG][NG / 2], int64_t k, int pos, int l) {
    if (a.src.scheme != SIGK_SCHEME_EXPLICIT) {
#pragma unroll
        for (int w = 0; w < NG; ++w)
#pragma unroll
            for (int h = 0; h < NG / 2; ++h)
                v[w][h] = make_float2(scheme_coef(v[w][h].x, a.src.scheme), scheme_coef(v[w][h].y, a.src.scheme));
    }
    kc_store<NG>(a.band, k, a.n_pairs, a.TperR, a.NQV, pos, l, v);
}

// Entry j of the staged column points as a pair (column, column - NG/2).
template <int NG>
__device__ __forceinline__ float2 kc_points(const float *q, int j) {
    if constexpr (kc_pp<NG>() == 2) return reinterpret_cast<const float2 *>(q)[j];
    else return make_float2(q[j], q[j - NG / 2]);
}

// The sums of a slot's first cells (RBF lift): rows h, h + NG/2 at entry NG - 1 -
// h of the column pairs (|u|^2, <u,dx>, <u,dy>), and row 0 in windows NG/2 + i and
// i at entry NG + NG/2 - 1 + i (<u,dy>).
template <int NG>
struct KcFirst {
    static constexpr int NH = NG / 2;
    float2 uu[NH], ux[NH], uy[NH], ur[NH];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int h = 0; h < NH; ++h) uu[h] = ux[h] = uy[h] = ur[h] = kc2(0.f);
    }
    // channel c: the lane's row points and increments, the columns' increments and points
    __device__ __forceinline__ void add(const float *xp, const float *xi, const float2 *e, const float *q, int l) {
        const float2 minus = kc2(-1.f);
        float2 xv[NH], dv[NH];
        kc_rows<NG>(xv, xp, l);
        kc_rows<NG>(dv, xi, l);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const float2 u = __ffma2_rn(kc_points<NG>(q, NG - 1 - h), minus, xv[h]);
            uu[h] = __ffma2_rn(u, u, uu[h]);
            ux[h] = __ffma2_rn(u, dv[h], ux[h]);
            uy[h] = __ffma2_rn(u, e[NG - 1 - h], uy[h]);
            const float2 t = __ffma2_rn(kc_points<NG>(q, NG + NH - 1 + h), minus, kc2(xv[0].x));
            ur[h] = __ffma2_rn(t, e[NG + NH - 1 + h], ur[h]);
        }
    }
};

// A slot that cannot be carried (RBF lift), formed one cell at a time: C and |u|^2 of
// every cell, and the exponents of its first ones (kc_exponents).
template <int NG>
struct KcRough {
    static constexpr int NH = NG / 2;
    float2 c[NG][NH], uu[NG][NH];
    float2 a[NH], b[NH], top[NH];
};
// A rough slot: the |u|^2 of its cells over the staged channels (xp, yp: the first
// one's), then their coefficients, to the band.  In a function of its own, so that
// the other slots' registers do not pay for it.  kappa comes from each cell's
// own distance; A and B move on by C, which costs them the rounding of a few
// additions.  A cell is the product form where A and B are below 1/2, else the
// difference of the two steps along the side that changes less (rbf.cuh), both
// for all, without branches; cells beside far jumps, where that rounding shows, are
// formed from their points.
template <int NG>
__device__ __noinline__ void kc_rough(KcRough<NG> &r, const KcArgs &a, const float *xp, const float *yp, int ys, int64_t k,
                                      int64_t row0, int64_t col0, int pos, int l) {
    constexpr int NH = NG / 2;
    const float2 minus = kc2(-1.f);
    {
        const int nc = (int)a.src.d;
        float2 uu[NG][NH];
#pragma unroll
        for (int w = 0; w < NG; ++w)
#pragma unroll
            for (int h = 0; h < NH; ++h) uu[w][h] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int c = 0; c < nc; ++c, xp += kc_xs<NG>(), yp += ys) {
            float2 xv[NH], yv[2 * NG - 1];
            kc_rows<NG>(xv, xp, l);
            if constexpr (NG == 8) {
                float q[16];
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                    const float4 t = *reinterpret_cast<const float4 *>(yp + j);
                    q[j] = t.x; q[j + 1] = t.y; q[j + 2] = t.z; q[j + 3] = t.w;
                }
#pragma unroll
                for (int j = NH; j < 2 * NG - 1; ++j) yv[j] = make_float2(q[j], q[j - NH]);
            } else {
#pragma unroll
                for (int j = NH; j < 2 * NG - 1; ++j) yv[j] = kc_points<NG>(yp, j);
            }
#pragma unroll
            for (int w = 0; w < NG; ++w)
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    const float2 u = __ffma2_rn(yv[NG - 1 + w - h], minus, xv[h]);
                    uu[w][h] = __ffma2_rn(u, u, uu[w][h]);
                }
        }
#pragma unroll
        for (int w = 0; w < NG; ++w)
#pragma unroll
            for (int h = 0; h < NH; ++h) r.uu[w][h] = uu[w][h];
    }
    const float s = a.s;
    float2 av[NH], bv[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) { av[h] = r.a[h]; bv[h] = r.b[h]; }
    float most = 0.f;   // the largest exponent so far
    auto exp2v = [](float2 v) { return make_float2(__expf(v.x), __expf(v.y)); };
    // a step of x from e0 to e1, series = e^x - 1 where |x| <= 1/2
    auto step = [](float x, float series, float e0, float e1) { return fabsf(x) <= 0.5f ? e0 * series : e1 - e0; };
#pragma unroll 1
    for (int w = 0; w < NG; ++w) {
        float2 an[NH];
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const float2 A = av[h], B = bv[h], C = r.c[w][h], E = __fmul2_rn(kc2(-s), r.uu[w][h]);
            const bool rx = fabsf(A.x) >= fabsf(B.x), ry = fabsf(A.y) >= fabsf(B.y);
            // v: the steps' exponent at this corner (the smaller one), o: between the two steps
            const float2 v = make_float2(rx ? B.x : A.x, ry ? B.y : A.y), o = make_float2(rx ? A.x : B.x, ry ? A.y : B.y);
            const float2 v1 = __fadd2_rn(v, C), E1 = __fadd2_rn(E, o);
            const float2 sv = kc_expm1<8>(v), so = kc_expm1<8>(o), sc = kc_expm1<8>(C), s1 = kc_expm1<8>(v1);
            const float2 e = exp2v(E), ev = exp2v(__fadd2_rn(E, v)), eo = exp2v(E1), eov = exp2v(__fadd2_rn(E1, v1));
            const float2 eC = __ffma2_rn(so, sc, sc);   // (1 + so) sc
            const float2 near = __fmul2_rn(e, __ffma2_rn(sv, so, __ffma2_rn(sv, eC, eC)));
            float2 c = near;
            if (fmaxf(fabsf(o.x), fabsf(C.x)) > 0.5f) c.x = step(v1.x, s1.x, eo.x, eov.x) - step(v.x, sv.x, e.x, ev.x);
            if (fmaxf(fabsf(o.y), fabsf(C.y)) > 0.5f) c.y = step(v1.y, s1.y, eo.y, eov.y) - step(v.y, sv.y, e.y, ev.y);
            // the exponents so far leave an error of their size times 2^-24; to the
            // points where it shows (a corner's kappa times it above 1e-7), or where
            // they are too large to tell
            most = fmaxf(most, fmaxf(fmaxf(fmaxf(fabsf(A.x), fabsf(A.y)), fmaxf(fabsf(B.x), fabsf(B.y))),
                                     fmaxf(fabsf(C.x), fabsf(C.y))));
            auto shows = [&](float E0, float top) {
                const float m = fmaxf(most, fabsf(E0));
                return m > 32.f && (m * top > 2.f || m > 1e7f);
            };
            const bool fx = shows(E.x, fmaxf(fmaxf(e.x, ev.x), fmaxf(eo.x, eov.x)));
            const bool fy = shows(E.y, fmaxf(fmaxf(e.y, ev.y), fmaxf(eo.y, eov.y)));
            if (fx || fy) {
                const int64_t d = a.src.d;
#pragma unroll 1
                for (int i = fx ? 0 : 1; i < (fy ? 2 : 1); ++i) {
                    const int g = h + i * NH, p = l * NG + g - a.vrows, q = pos * NG + w - g - a.NQV;
                    float t = 0.f;
                    if (p >= 0 && q >= 0 && q < (int)a.src.Lb - 1)
                        t = rbf_far_cell((const float *)a.src.A + (row0 + p) * d,
                                         (const float *)a.src.B + (col0 + q) * d, d, s);
                    if (i == 0) c.x = t;
                    else c.y = t;
                }
            }
            r.c[w][h] = __fmul2_rn(kc2(a.scale), c);
            an[h] = __fadd2_rn(A, C);
            bv[h] = __fadd2_rn(B, C);
        }
#pragma unroll
        for (int h = NH - 1; h >= 1; --h) av[h] = an[h - 1];
        av[0] = make_float2(w + 1 < NH ? r.top[w + 1].y : w + 1 < NG ? r.top[w + 1 - NH].x : 0.f, an[NH - 1].x);
    }
    kc_put<NG>(a, r.c, k, pos, l);
}

// A slot's sums <dx,dy> into its coefficients (RBF lift).  Everything is done
// for rows h and h + NG/2 at once; at window w row g is one column ahead of row
// g + 1, so a(g + 1) of the next window is a(g) + (1 + a(g)) e(g) of this one.
// False where the slot is rough: r then holds its C's and first exponents.
template <int NG>
__device__ __forceinline__ bool kc_lift(float2 (&acc)[NG][NG / 2], const KcFirst<NG> &first, KcRough<NG> &r,
                                        const KcArgs &a, int l, const float *xx, const float *yy) {
    constexpr int NH = NG / 2;
    const float s = a.s, s2 = 2.f * s;
    float far = 0.f;
#pragma unroll
    for (int w = 0; w < NG; ++w)
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            acc[w][h] = __fmul2_rn(acc[w][h], kc2(s2));   // C
            far = fmaxf(far, fmaxf(fabsf(acc[w][h].x), fabsf(acc[w][h].y)));
        }
    far *= NG;
    float2 av[NH], bv[NH], kap[NH], top[NH], sq[NH];
    kc_rows<NG>(sq, xx, l);
    auto arg = [&](float2 sum, float2 sqr, float sign) {   // sign s (2 sum + sign' square), its size noted
        const float2 v = __fmul2_rn(kc2(sign * s), __ffma2_rn(kc2(2.f), sum, __fmul2_rn(kc2(-sign), sqr)));
        far = fmaxf(far, fmaxf(fabsf(v.x), fabsf(v.y)));
        return v;
    };
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        av[h] = arg(first.uy[h], make_float2(yy[NG - 1 - h], yy[NH - 1 - h]), 1.f);
        top[h] = arg(first.ur[h], make_float2(yy[NG + NH - 1 + h], yy[NG - 1 + h]), 1.f);
        bv[h] = arg(first.ux[h], sq[h], -1.f);
    }
    if (far > KC_CARRY) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            r.a[h] = av[h];
            r.b[h] = bv[h];
            r.top[h] = top[h];
        }
#pragma unroll
        for (int w = 0; w < NG; ++w)
#pragma unroll
            for (int h = 0; h < NH; ++h) r.c[w][h] = acc[w][h];
        return false;
    }
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        av[h] = kc_expm1<8>(av[h]);
        bv[h] = kc_expm1<8>(bv[h]);
        top[h] = kc_expm1<8>(top[h]);
        kap[h] = make_float2(a.scale * __expf(-s * first.uu[h].x), a.scale * __expf(-s * first.uu[h].y));
    }
#pragma unroll
    for (int w = 0; w < NG; ++w) {
        float2 an[NH];
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const float2 e = kc_expm1<NG == 8 ? 5 : NG == 4 ? 6 : 7>(acc[w][h]);
            const float2 ea = __ffma2_rn(av[h], e, e), eb = __ffma2_rn(bv[h], e, e);
            acc[w][h] = __fmul2_rn(kap[h], __ffma2_rn(av[h], bv[h], __ffma2_rn(bv[h], ea, ea)));
            kap[h] = __ffma2_rn(kap[h], av[h], kap[h]);
            an[h] = __fadd2_rn(av[h], ea);
            bv[h] = __fadd2_rn(bv[h], eb);
        }
        // row g + 1 takes row g's; row 0 its own of the next column
#pragma unroll
        for (int h = NH - 1; h >= 1; --h) av[h] = an[h - 1];
        av[0] = make_float2(w + 1 < NH ? top[w + 1].y : w + 1 < NG ? top[w + 1 - NH].x : 0.f, an[NH - 1].x);
    }
    return true;
}

// MULTI: more channels than are staged at once (one pass; linear kernel)
template <int NG, bool RBF, bool MULTI>
__global__ void __launch_bounds__(KcShape<NG, RBF>::WARPS * 32, KcShape<NG, RBF>::MINB) band_coef_kernel(KcArgs a) {
    extern __shared__ __align__(16) float kc_sm[];
    constexpr int NPP = 32 * NG, XS = kc_xs<NG>(), NP = KcShape<NG, RBF>::NP, NH = NG / 2;
    using Sh = KcShape<NG, RBF>;
    const int nt = blockDim.x, tid = threadIdx.x, warp = tid >> 5;
    const int lw = tid & (Sh::LW - 1), jw = (tid & 31) / Sh::LW;   // lane and position in the warp's item
    const int64_t d = a.src.d;
    const int nch = RBF || d < KC_CH ? (int)d : KC_CH, YS = kc_ys(a.tp, NG);
    float *xi = kc_sm;                                            // row increments (linear: scaled)
    float *y0 = xi + a.xch * XS;                                  // the next step's column points
    float2 *yi = reinterpret_cast<float2 *>(y0 + nch * YS);       // pairs of column increments
    float *yp = reinterpret_cast<float *>(yi + nch * YS);         // RBF: this step's column points,
    float *xp = yp + nch * YS * kc_pp<NG>();                      // row points, and the squared
    float *xx = xp + a.xch * XS, *yy = xx + XS;                   // increments of rows and columns
    const int64_t units = a.n_pairs * a.tiles, per = (units + gridDim.x - 1) / gridDim.x;
    const int64_t ubeg = (int64_t)blockIdx.x * per;
    const int64_t uend = ubeg + per < units ? ubeg + per : units;
    if (ubeg >= uend) return;
    const int ny = (int)a.src.Lb - 1;
    const bool keep = !MULTI || a.xch == (int)d;   // all of a row path's channels stay
    const int chunks = MULTI ? a.chunks : 1, passes = MULTI ? 1 : a.passes;

    // channels c0 .. c0 + nc - 1 of the row path's increments (and points) from xi[at XS] on
    auto stage_x = [&](int64_t row0, int64_t c0, int nc, int at) {
        const float *x = (const float *)a.src.A + row0 * d + c0;
        const int gs = kc_group(nc);
        for (int c = tid & (gs - 1); c < nc; c += RBF ? gs : nc)
            for (int P = tid / gs; P < NPP; P += nt / gs) {
                const int p = P - a.vrows;
                const float *r = x + (int64_t)(p < 0 ? 0 : p) * d + c;
                const float e = p >= 0 ? __ldg(r + d) - __ldg(r) : 0.f;
                xi[(at + c) * XS + kc_xpos<NG>(P)] = RBF ? e : e * a.scale;
                if (RBF) xp[(at + c) * XS + kc_xpos<NG>(P)] = __ldg(r);
            }
    };
    // tile t's column points, ends repeated, into y0[c][iq], Q = t tp NG + iq - (NG - 1)
    auto fetch_y = [&](int64_t row0, int t, int64_t c0, int nc) {
        const float *y = (const float *)a.src.B + row0 * d + c0;
        const int gs = kc_group(nc), Q0 = t * a.tp * NG - (NG - 1) - a.NQV;
        for (int c = tid & (gs - 1); c < nc; c += RBF ? gs : nc)
            for (int iq = tid / gs; iq < YS; iq += nt / gs) {
                int q = Q0 + iq;
                q = q < 0 ? 0 : (q > ny ? ny : q);
                kc_cp4(y0 + c * YS + iq, y + (int64_t)q * d + c);
            }
        kc_commit();
    };
    // the pairs (column iq, column iq - NG/2) from the fetched points; RBF: and the
    // squared increments, over the channels so far (rows': of the xc staged from c0)
    auto pair_y = [&](int64_t c0, int nc, int xc) {
        for (int iq = tid; iq < YS; iq += nt) {
            float sq = RBF && c0 > 0 ? yy[iq] : 0.f;
            const int ib = iq >= NH ? iq - NH : 0, hi = iq + 1 < YS ? 1 : 0;
            for (int c = 0; c < nc; ++c) {
                const float *y = y0 + c * YS;
                const float ya = y[iq], yb = y[ib];
                const float2 e = make_float2(y[iq + hi] - ya, y[ib + 1] - yb);
                yi[c * YS + iq] = e;
                if (RBF) {
                    if constexpr (kc_pp<NG>() == 2)
                        reinterpret_cast<float2 *>(yp)[c * YS + iq] = make_float2(ya, yb);
                    else
                        yp[c * YS + iq] = ya;
                    sq = fmaf(e.x, e.x, sq);
                }
            }
            if (RBF) yy[iq] = sq;
        }
        if (RBF && xc > 0)
            for (int P = tid; P < NPP; P += nt) {
                float sq = c0 > 0 ? xx[P] : 0.f;
                for (int c = 0; c < xc; ++c) sq = fmaf(xi[c * XS + P], xi[c * XS + P], sq);
                xx[P] = sq;   // in the staged order, as xi
            }
    };

    int64_t kn = ubeg / a.tiles;          // the next step's pair and tile
    int tn = (int)(ubeg - kn * a.tiles);
    PairRef pr = pair_ref<true>(a.src, kn);
    int64_t staged = -1;   // the row path whose values xi (and xp) hold
    fetch_y(pr.b_row0, tn, 0, nch);
    float2 acc[NP][NG][NH];
    for (int64_t u = ubeg; u < uend; ++u) {
        const PairRef cur = pr;
        const int64_t k = kn;
        const int t = tn;
        const bool more = u + 1 < uend;
        if (more && ++tn == a.tiles) {
            tn = 0;
            pr = pair_ref<true>(a.src, ++kn);
        }
        for (int ch = 0; ch < chunks; ++ch) {
            const int64_t c0 = (int64_t)ch * KC_CH;
            const int nc = RBF ? (int)d : d - c0 < KC_CH ? (int)(d - c0) : KC_CH;
            kc_wait();
            __syncthreads();   // this step's columns are here, and the last step's readers are done
            const bool fresh = !keep || staged != cur.a_row0;
            if (fresh) {
                if (keep)
                    for (int64_t c = 0; c < d; c += RBF ? d : KC_CH)
                        stage_x(cur.a_row0, c, RBF ? (int)d : d - c < KC_CH ? (int)(d - c) : KC_CH, (int)c);
                else
                    stage_x(cur.a_row0, c0, nc, 0);
                staged = cur.a_row0;
                if (RBF) __syncthreads();
            }
            pair_y(c0, nc, !fresh ? 0 : keep ? (int)d : nc);
            __syncthreads();
            if (ch + 1 < chunks) fetch_y(cur.b_row0, t, c0 + KC_CH, d - c0 - KC_CH < KC_CH ? (int)(d - c0 - KC_CH) : KC_CH);
            else if (more) fetch_y(pr.b_row0, tn, 0, nch);
            const float *xc = xi + (keep ? (int)c0 * XS : 0), *xq = xp + (keep ? (int)c0 * XS : 0);
            for (int pass = 0; pass < passes; ++pass) {
                // the warp's item: a block of lanes and a group of positions
                const int item = pass * (nt >> 5) + warp, l = item % (32 / Sh::LW) * Sh::LW + lw;
                const int off = item / (32 / Sh::LW) * Sh::GP + jw * NP;
                const bool live = off < a.tp && t * a.tp + off <= a.TperR;
                const int rel = live ? off : 0, pos = t * a.tp + rel;
                if (ch == 0) {
#pragma unroll
                    for (int n = 0; n < NP; ++n)
#pragma unroll
                        for (int w = 0; w < NG; ++w)
#pragma unroll
                            for (int h = 0; h < NH; ++h) acc[n][w][h] = make_float2(0.f, 0.f);
                }
                const float2 *yr = yi + rel * NG;   // entry j: columns Q = pos NG - (NG - 1) + j and Q - NG/2
#pragma unroll 2
                for (int c = 0; c < nc; ++c) {
                    float2 xv[NH], yv[(NP + 1) * NG - NH];
                    kc_rows<NG>(xv, xc + c * XS, l);
                    kc_cols<NG>(yv, yr + c * YS + NH);
#pragma unroll
                    for (int n = 0; n < NP; ++n)
#pragma unroll
                        for (int w = 0; w < NG; ++w)
#pragma unroll
                            for (int h = 0; h < NH; ++h)
                                acc[n][w][h] = __ffma2_rn(xv[h], yv[n * NG + w - h + NG - 1 - NH], acc[n][w][h]);
                }
                auto add_first = [&](KcFirst<NG> &f, int n) {
#pragma unroll 1
                    for (int c = 0; c < nc; ++c)
                        f.add(xq + c * XS, xc + c * XS, yr + c * YS + n * NG,
                              yp + (c * YS + (rel + n) * NG) * kc_pp<NG>(), l);
                };
                if (!live || ch + 1 < chunks) continue;
                KcRough<NG> rough[RBF ? NP : 1];
                unsigned bad = 0;   // the slots that are rough
#pragma unroll
                for (int n = 0; n < NP; ++n) {
                    if (n > 0 && (rel + n >= a.tp || pos + n > a.TperR)) break;
                    if constexpr (RBF) {
                        KcFirst<NG> f;
                        f.clear();
                        add_first(f, n);
                        if (!kc_lift<NG>(acc[n], f, rough[n], a, l, xx, yy + (rel + n) * NG)) {
                            bad |= 1u << n;
                            continue;
                        }
                    }
                    kc_put<NG>(a, acc[n], k, pos + n, l);
                }
                if constexpr (RBF) {
                    if (bad)
#pragma unroll 1
                        for (int n = 0; n < NP; ++n)
                            if (bad >> n & 1)
                                kc_rough<NG>(rough[n], a, xq, yp + (rel + n) * NG * kc_pp<NG>(), YS * kc_pp<NG>(), k,
                                             cur.a_row0, cur.b_row0, pos + n, l);
                }
            }
        }
    }
}

template <int NG, bool RBF>
cudaError_t launch(const KcArgs &a0, int sms, cudaStream_t st) {
    KcArgs a = a0;
    const int npos = a.TperR + 1;
    using Sh = KcShape<NG, RBF>;
    const int d = (int)a.src.d, nch = RBF || d < KC_CH ? d : KC_CH;
    a.chunks = (d + nch - 1) / nch;
    // the largest even share of the positions that fits
    auto share = [&](int most) {
        a.tiles = (npos + most - 1) / most;
        a.tp = ((npos + a.tiles - 1) / a.tiles + Sh::NP - 1) / Sh::NP * Sh::NP;
        return (int)sizeof(float) * kc_smem_floats<NG, RBF>(a.tp, nch, nch) <= SMEM_LIMIT;
    };
    for (int most = a.chunks > 1 ? Sh::TILEC : Sh::TILE; !share(most); most -= Sh::GP) {}
    // a row path's channels all stay where they fit (two chunks do)
    a.xch = d;
    int smem = (int)sizeof(float) * kc_smem_floats<NG, RBF>(a.tp, nch, nch);
    if (d <= 4 * KC_CH && (int)sizeof(float) * kc_smem_floats<NG, RBF>(a.tp, nch, d) <= SMEM_LIMIT)
        smem = (int)sizeof(float) * kc_smem_floats<NG, RBF>(a.tp, nch, d);
    else
        a.xch = nch;
    const int items = (a.tp + Sh::GP - 1) / Sh::GP * (32 / Sh::LW);
    const int most = RBF && NG < 8 && smem <= SMEM_LIMIT / 2 ? Sh::WARPS / 2 : Sh::WARPS;
    a.passes = a.chunks > 1 ? 1 : (items + most - 1) / most;
    const int warps = (items + a.passes - 1) / a.passes;
    auto go = [&](auto kern) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, warps * 32, smem)) != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        int64_t grid = (int64_t)sms * per_sm;
        if (grid > a.n_pairs * a.tiles) grid = a.n_pairs * a.tiles;
        kern<<<(int)grid, warps * 32, smem, st>>>(a);
        return cudaGetLastError();
    };
    if constexpr (!RBF)
        if (a.chunks > 1) return go(band_coef_kernel<NG, false, true>);
    return go(band_coef_kernel<NG, RBF, false>);
}

// The band as rbf.cuh's tiles write it: coarse cell (p, q) is the padded cell (P, Q)
// = (p + vrows, q + NQV), in lane P / NG as row g = P % NG, at the position pos and
// window w with pos NG + w = Q + g.
template <int NG>
struct KcTileLayout {
    PairSrc src;
    float *band;
    int64_t nslots;
    int TperR, NQV, vrows;
    struct Geo {
        const float *rows, *cols;
        int nx, ny;
        int64_t k;
    };
    struct Row {
        int l, g;
    };
    __device__ Geo geo(int64_t k) const {
        const PairRef pr = pair_ref<true>(src, k);
        return {(const float *)src.A + pr.a_row0 * src.d, (const float *)src.B + pr.b_row0 * src.d, (int)pr.la - 1,
                (int)pr.lb - 1, k};
    }
    __device__ Row row(const Geo &, int p) const { return {(p + vrows) / NG, (p + vrows) % NG}; }
    __device__ void store(const Geo &g, const Row &r, int q, float c) const {
        const int t = q + NQV + r.g, at = t % NG * NG + 2 * (r.g % (NG / 2)) + r.g / (NG / 2);
        band[band_row(g.k * TperR + t / NG, r.l, NG, nslots) + band_off(at)] = c;
    }
};

template <int NG>
cudaError_t launch_tiles(const KcArgs &a, int sms, cudaStream_t st) {
    const int64_t nslots = a.n_pairs * a.TperR + 1;
    const KcTileLayout<NG> lay = {a.src, a.band, nslots, a.TperR, a.NQV, a.vrows};
    return launch_rbf_coef<float>(lay, a.n_pairs, a.src.La - 1, a.src.Lb - 1, a.src.d, a.src.sigma, (double)a.scale,
                                  a.src.scheme, a.band, sizeof(float) * (size_t)nslots * 32 * NG * NG, sms, st);
}

// The lift with more channels than a block stages takes rbf.cuh's tiles, every cell
// from its own six sums.  Carrying over several passes of channels keeps twice the
// sums in registers: 1.07 times as fast as the tiles at d = 130 (48 x 48 paths of 100
// and 90 points, order 1), 0.67 times at d = 100 (96 x 96 of 30 and 33, order 0), and
// on rough data, where a slot needs every channel once more, a third to a half.  With
// all of d = 64 staged at once it is 1.4 times as fast (64 x 64 of 128, order 0).
constexpr int KC_LIFT = 64;

}  // namespace

cudaError_t launch_band_coefs(const PairSrc &src, const BandPlan &p, int64_t n_pairs, float *band, int sms,
                              cudaStream_t st) {
    KcArgs a;
    a.src = src;
    a.band = band;
    a.n_pairs = n_pairs;
    a.TperR = p.TperR;
    a.NQV = p.NQV;
    a.vrows = p.vrows;
    a.tiles = a.tp = a.passes = a.chunks = a.xch = 1;
    a.scale = 0.5f / (float)(1 << (2 * p.lam));
    a.s = (float)(0.5 / (src.sigma * src.sigma));
    const bool rbf = src.kernel == SIGK_KERNEL_RBF;
    if (rbf && src.d > KC_LIFT)
        return p.NG == 8 ? launch_tiles<8>(a, sms, st)
                         : p.NG == 4 ? launch_tiles<4>(a, sms, st) : launch_tiles<2>(a, sms, st);
    if (p.NG == 8) return rbf ? launch<8, true>(a, sms, st) : launch<8, false>(a, sms, st);
    if (p.NG == 4) return rbf ? launch<4, true>(a, sms, st) : launch<4, false>(a, sms, st);
    return rbf ? launch<2, true>(a, sms, st) : launch<2, false>(a, sms, st);
}

}  // namespace sigk
