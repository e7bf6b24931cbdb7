// Forward sweep, FP32, "band" form: the row-chain wavefront of fwd_chain.cu
// (one warp solves a chain of pairs of equal shape, lane l owning refined rows
// R*l .. R*l+R-1, the difference form Q(a,b) = Q(a-1,b) + c (K(a,b-1) +
// K(a-1,b)), K(a,b) = K(a,b-1) + Q(a,b) of the scheme of Sec. 3.1), with the
// coarse-cell coefficients c = 1/2 4^-lambda <dx_p, dy_q> (remark after the
// scheme) formed beforehand by a contraction kernel instead of inside the
// sweep.  That pays off when d is large: the sweep costs 3 operations per
// refined cell, an inline dot product d / 4^lambda more.
//
// The coefficient buffer is laid out for the sweep ("band" layout).  In
// macro-step pos of a pair (columns pos*NG .. pos*NG + NG - 1 of the padded
// coarse grid, NG = R / 2^lambda coarse rows per lane), window w, group g of
// lane l is at coarse cell (P, Q) = (l*NG + g, pos*NG + w - g).  Slot (pair,
// pos, lane) holds these NG x NG values as [w][g]; where its elements lie:
// band_row, band_off.  Cells with Q < 0 (pos = 0, w < g) are the previous pair's
// last columns, which rows that have not turned over yet still need: they are
// stored in the next pair's slot 0, so the chain reads pair k's coefficients,
// tail included, from slots (k, 0 .. TperR - 1) and (k + 1, 0).  Virtual rows
// and columns (padding, as in fwd_chain.cu) hold 0.  What the sweeps write per
// cell (dk/dc, the surface's nodes) goes to the same slots, TperR + 1 a pair,
// each lane's kept whole ([pair][pos][lane][w][g]).
#include <string.h>

#include <type_traits>

#include "sigk_internal.cuh"
#include "tc5.cuh"
#include "tile_gemm.cuh"

namespace sigk {

namespace {

constexpr int BAND_WARPS = 2;   // warps per CTA of the sweep

struct BandCoefArgs {
    PairSrc src;
    int64_t n_pairs;      // pairs of this launch (slot rows 0 .. n_pairs)
    int TperR, NQ, NQV, vrows;
    float scale;          // 1/2 4^-lambda
    float *band;
};

// Order of the groups inside a window of a slot: g and g + NG/2 side by side
// (the sweeps carry groups g and g + NG/2 as one float2).
template <int NG>
__host__ __device__ constexpr int band_gpos(int g) {
    return g < NG / 2 ? 2 * g : 2 * (g - NG / 2) + 1;
}

struct BandArgs {
    PairSrc src;
    float *out;
    const float *band;
    int64_t n_pairs, ppw;
    int TperR;
    // what the adjoint needs to run the sweep backwards (null: forward only)
    float *ckpt;     // [warp][nck][lane][2R]: (K, Q) of every row after each BAND_CK-th macro-step
    float *exitk;    // [pair][lane][R]: K of each row on its pair's last column
    float *botq;     // [warp][steps + 1]: Q of the warp's last row before each step
    int nck;         // checkpoint slots per warp
    int64_t bq_stride;
    // the solution surface on the sample grid (SURF instances): each lane's
    // values at the sample-grid nodes, a window row per window, in the band
    // layout with TperR + 1 slots per pair (slot TperR: the tail); unpacked by
    // band_gbar_kernel in surface mode
    float *sband;
};

constexpr int BAND_CK = 8;   // macro-steps between checkpoints of the forward state

// Window w of the slot at p (band_row).
template <int NG>
__device__ __forceinline__ void load_window(float (&v)[NG], const float *slot, int w) {
    const float *p = slot + band_off(w * NG);
    if constexpr (NG == 8) {
        const float4 a = __ldcs(reinterpret_cast<const float4 *>(p));
        const float4 b = __ldcs(reinterpret_cast<const float4 *>(p + 128));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else if constexpr (NG == 4) {
        const float4 a = __ldcs(reinterpret_cast<const float4 *>(p));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    } else {
        const float2 a = __ldcs(reinterpret_cast<const float2 *>(p));
        v[0] = a.x; v[1] = a.y;
    }
}

// A window row of NG values (NH float2: groups g, g + NH) to 16-byte aligned
// band memory.
template <int NG>
__device__ __forceinline__ void store_window(float *dst, const float2 (&v)[NG / 2]) {
    if constexpr (NG == 8) {
        reinterpret_cast<float4 *>(dst)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        reinterpret_cast<float4 *>(dst)[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
    } else if constexpr (NG == 4) {
        reinterpret_cast<float4 *>(dst)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    } else {
        reinterpret_cast<float2 *>(dst)[0] = v[0];
    }
}

// Macro-steps of coefficients in flight per warp, by cp.async into shared memory,
// where a macro-step is too short (R < 16 steps) for a load issued one ahead
// to arrive in time: 32 steps' worth.  0: registers, refilled window by window
// a macro-step ahead (R = 16, and the 8 KB slots of R = NG = 8).  24 x 17 paths of
// 50 and 71 points, order 1 (R = 4): the checkpointing sweep 90 -> 18 us, the
// adjoint 72 -> 49 us.
template <int R, int NG>
__host__ __device__ constexpr int band_ring() { return R < 16 && NG <= 4 ? 32 / R : 0; }

template <int NBYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (NBYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(NBYTES) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// The sweep: fwd_chain.cu's chain_f32_kernel with its staging and dot
// products replaced by one coefficient vector per window, prefetched one
// macro-step ahead into the registers the window has just consumed.
//
// SURF: also keep the solution at the sample-grid nodes (the surface).  Row
// r of lane l, padded row R l + r, is refined node row a = R l + r + 1 - vtop;
// at step j of position pos it computes padded column pos R + j - r (the
// previous pair's when negative), node column b = that + 1 - vpad.  vtop and
// vpad are multiples of 2^lambda, so the node is on the sample grid exactly
// when a and b are: r % 2^lambda = 2^lambda - 1 (the last row of each coarse
// group), and then b = j - r + 1 = j + 2 (mod 2^lambda), i.e. at step
// j % 2^lambda = 2^lambda - 2 of each window (0 for dyadic orders 0 and 1).
// There, group g of window w holds node (p + 1, q) (dyadic order 0: (p + 1,
// q + 1)) of the coarse cell (p, q) = (P - vrows, Q - NQV), (P, Q) = (lane NG
// + g, pos NG + w - g): the band layout's cell, so the lane stores its NG
// values as one window row.
template <int R, int LAM, int MINB, bool SAVE, bool SURF = false>
__global__ void __launch_bounds__(BAND_WARPS * 32, MINB) chain_band_kernel(BandArgs a) {
    constexpr int S = 1 << LAM;
    constexpr int NG = R / S;
    constexpr int H = R / 2;
    constexpr int NH = NG / 2;
    constexpr int JOUT = R - 2;
    constexpr int SLOT = NG * NG;
    static_assert(R % S == 0 && NG % 2 == 0 && NG <= 8, "2, 4 or 8 coarse rows per lane");

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int64_t gw = (int64_t)blockIdx.x * BAND_WARPS + warp;
    const int64_t k0 = gw * a.ppw;
    if (k0 >= a.n_pairs) return;   // whole warp
    const int np = (int)min(a.ppw, a.n_pairs - k0);
    const int TperR = a.TperR;

    float2 KP[H], QP[H];
    float2 CN[NH], CO[NH];
    float cb[NG][NG];   // this macro-step's coefficients [window][group]; refilled window by window
#pragma unroll
    for (int i = 0; i < H; ++i) { KP[i] = make_float2(1.f, 1.f); QP[i] = make_float2(0.f, 0.f); }
#pragma unroll
    for (int g = 0; g < NH; ++g) { CN[g] = make_float2(0.f, 0.f); CO[g] = CN[g]; }
    float pK = 1.f, pQ = 0.f;

    // the lane's slot in macro-step m (linear position m - lane of the chain), or
    // null outside the chain (its first pair's rows before they start, and after
    // the last pair except the slot that holds that pair's tail)
    const int64_t nslots = a.n_pairs * TperR + 1;
    auto slot = [&](int64_t m) -> const float * {
        return m >= lane && m - lane <= (int64_t)np * TperR
                   ? a.band + band_row(k0 * TperR + m - lane, lane, NG, nslots) : nullptr;
    };
    constexpr int D = band_ring<R, NG>();
    __shared__ __align__(16) float ring[D ? BAND_WARPS * D * 32 * SLOT : 1];
    float *rw = ring + (D ? warp * D * 32 * SLOT : 0) + 4 * lane;
    auto fetch = [&](int64_t m) {   // into the ring, quads of a lane 128 floats apart as in the band
        const float *p = slot(m);
        float *dst = rw + (int)(m % (D ? D : 1)) * 32 * SLOT;
#pragma unroll
        for (int i = 0; i < SLOT; i += 4) {
            if (p) cp_async<16>(dst + band_off(i), p + band_off(i));
            else *reinterpret_cast<float4 *>(dst + band_off(i)) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        cp_commit();
    };

    int kl = (lane == 0) ? 0 : -((lane + TperR - 1) / TperR);
    int pos = -lane - kl * TperR;
    if constexpr (D > 0) {
#pragma unroll
        for (int m = 0; m < D - 1; ++m) fetch(m);
    } else {
        const float *p0 = slot(0);
#pragma unroll
        for (int w = 0; w < NG; ++w) {
            if (p0) load_window<NG>(cb[w], p0, w);
            else
#pragma unroll
                for (int g = 0; g < NG; ++g) cb[w][g] = 0.f;
        }
    }
    const int64_t total_m = (int64_t)np * TperR + 32;
    float *bq = SAVE ? a.botq + gw * a.bq_stride : nullptr;
    if (SAVE && lane == 31) bq[0] = 0.f;

    for (int64_t m = 0; m < total_m; ++m) {
        const bool trans = (pos == 0);
        const float *pn = nullptr;
        if constexpr (D > 0) {
            fetch(m + D - 1);
            cp_wait<D - 1>();   // macro-step m's have landed
            const float *src = rw + (int)(m % D) * 32 * SLOT;
#pragma unroll
            for (int i = 0; i < SLOT; i += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(src + band_off(i));
                cb[i / NG][i % NG] = v.x;
                cb[(i + 1) / NG][(i + 1) % NG] = v.y;
                cb[(i + 2) / NG][(i + 2) % NG] = v.z;
                cb[(i + 3) / NG][(i + 3) % NG] = v.w;
            }
        } else {
            pn = slot(m + 1);
        }
        // exit states go to the pair the rows leave (kl - 1), when it is one of the chain's
        float *ex = (SAVE && trans && kl >= 1 && kl <= np)
                        ? a.exitk + ((k0 + kl - 1) * 32 + lane) * (int64_t)R : nullptr;

#pragma unroll
        for (int w = 0; w < NG; ++w) {
#pragma unroll
            for (int g = 0; g < NH; ++g) {
                CO[g] = CN[g];
                CN[g] = make_float2(cb[w][2 * g], cb[w][2 * g + 1]);   // groups g, g + NH
            }
            if constexpr (D == 0) {
                if (pn) load_window<NG>(cb[w], pn, w);
                else
#pragma unroll
                    for (int g = 0; g < NG; ++g) cb[w][g] = 0.f;
            }
#pragma unroll
            for (int jj = 0; jj < S; ++jj) {
                const int j = w * S + jj;
                const float kH1 = KP[H - 1].x, qH1 = QP[H - 1].x;   // row H-1 before this step
                float shK = 0.f, shQ = 0.f;
#pragma unroll
                for (int i = H - 1; i >= 0; --i) {
                    const int g1 = i / S, s1 = i % S;   // row i; row i+H: group g1+NH, same s1
                    if (jj == s1 && trans) {            // row starts its next pair now: k(.,0) = 1
                        if (g1 == w) {
                            if (ex) ex[i] = KP[i].x;
                            KP[i].x = 1.f;
                        }
                        if (g1 + NH == w) {
                            if (ex) ex[i + H] = KP[i].y;
                            KP[i].y = 1.f;
                        }
                    }
                    const float2 c = (jj >= s1) ? CN[g1] : CO[g1];
                    float2 ku, qu;
                    if (i > 0) {
                        ku = KP[i > 0 ? i - 1 : 0];
                        qu = QP[i > 0 ? i - 1 : 0];
                    } else {
                        ku = make_float2(pK, kH1);
                        qu = make_float2(pQ, qH1);
                    }
                    const float2 sum = __fadd2_rn(KP[i], ku);
                    const float2 qn = __ffma2_rn(c, sum, qu);
                    KP[i] = __fadd2_rn(KP[i], qn);
                    QP[i] = qn;
                    if (i == H - 1) {
                        shK = __shfl_up_sync(FULL, KP[i].y, 1);
                        shQ = __shfl_up_sync(FULL, QP[i].y, 1);
                        if (j == JOUT && trans && lane == 31) {
                            const int kp = kl - 1;   // row R-1 just finished pair kp's last column
                            if (kp >= 0 && kp < np && a.out) {
                                const PairRef pr = pair_ref<true>(a.src, k0 + kp);
                                a.out[pr.out0] = KP[i].y;
                                if (pr.out1 >= 0) a.out[pr.out1] = KP[i].y;
                            }
                        }
                    }
                }
                if constexpr (SURF) {
                    constexpr int JS = S >= 2 ? S - 2 : 0;
                    if (jj == JS) {
                        // rows g S + S - 1 (packed with g + NH) are at their group's node
                        float2 sv[NH];
#pragma unroll
                        for (int g = 0; g < NH; ++g) sv[g] = KP[g * S + S - 1];
                        if (kl >= 0 && kl < np)
                            store_window<NG>(a.sband + (((k0 + kl) * (TperR + 1) + pos) * 32 + lane) * (int64_t)SLOT +
                                                 w * NG, sv);
                        if (trans && kl >= 1 && kl <= np)   // the previous pair's tail
                            store_window<NG>(a.sband + (((k0 + kl - 1) * (TperR + 1) + TperR) * 32 + lane) *
                                                           (int64_t)SLOT + w * NG, sv);
                    }
                }
                if (SAVE && lane == 31) bq[m * R + j + 1] = QP[H - 1].y;
                pK = (lane == 0) ? 1.f : shK;
                pQ = (lane == 0) ? 0.f : shQ;
            }
        }
        if (SAVE && ((m + 1) % BAND_CK == 0 || m == total_m - 1)) {
            float4 *ck = reinterpret_cast<float4 *>(a.ckpt + ((gw * a.nck + m / BAND_CK) * 32 + lane) * (int64_t)(2 * R));
#pragma unroll
            for (int i = 0; i < H; i += 2) {
                ck[i / 2] = make_float4(KP[i].x, KP[i].y, KP[i + 1].x, KP[i + 1].y);
                ck[H / 2 + i / 2] = make_float4(QP[i].x, QP[i].y, QP[i + 1].x, QP[i + 1].y);
            }
        }
        if (++pos == TperR) {
            pos = 0;
            ++kl;
        }
    }
    if constexpr (D > 0) cp_wait<0>();
}

// The band's coefficients on the fifth-generation tensor cores (tcgen05), for d <= 64.
// A block takes a contiguous run of pairs; per pair, per 128-row tile of the
// padded rows: the row increments (scaled by 1/2 4^-lambda) are split into
// TF32 hi and lo parts and staged once, then the padded columns are walked in
// chunks of 128 (the next chunk's increments fetched while the MMAs run): one
// thread issues the split-TF32 MMA chain (D = 128 x 128 fp32 in TMEM), the
// warps copy D into a shared tile, and each warp then writes four slot
// positions of one lane block, lane (s, g) reading row l*NG + g of the tile
// along the slot's window (conflict-free with the tile stride 132) and the
// lanes of a slot storing one 32-byte window row together.  Entries outside
// the chunk, and the previous pair's cells of slot 0, are left to the chunk or
// pair that owns them; the pair's tail goes to slot 0 of the next pair.  Waits
// are bounded (status word SIGK_ETIMEOUT).
constexpr int BT5_M = 128, BT5_N = 128, BT5_SS = BT5_N + 4, BT5_T = 256;

inline int bt5_smem_bytes(int64_t d) { return 4 * BT5_M * tc5::tc5_k_of(d) * 4 + BT5_M * BT5_SS * 4; }

template <int NG>
__global__ void __launch_bounds__(BT5_T, 1) band_coef_tc5_kernel(BandCoefArgs a, int *status, long long max_wait) {
    constexpr int SLOT = NG * NG;
    constexpr int NPP = 32 * NG;          // padded rows
    constexpr int SPW = 32 / NG;          // slot positions per warp task (lane = s * NG + g)
    extern __shared__ __align__(1024) unsigned char bt5_sm[];
    __shared__ __align__(8) unsigned long long mbar;
    __shared__ unsigned tmem_slot;
    const int64_t d = a.src.d;
    const int K = tc5::tc5_k_of(d);
    const int D4 = (int)((d + 3) / 4);
    unsigned char *ah = bt5_sm, *al = ah + BT5_M * K * 4;
    unsigned char *bh = al + BT5_M * K * 4, *bl = bh + BT5_N * K * 4;
    float *St = reinterpret_cast<float *>(bl + BT5_N * K * 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = tid & (BT5_M - 1), half = tid >> 7;
    const unsigned idesc = tc5::idesc_tf32(BT5_M, BT5_N);
    const int TperR = a.TperR, NQ = a.NQ;

    if (warp == 0) tc5::alloc(&tmem_slot, BT5_N);
    if (tid == 0) tc5::mbar_init(&mbar);
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    const unsigned tmem = tmem_slot;
    unsigned phase = 0;
    bool failed = false;

    const int64_t per = (a.n_pairs + gridDim.x - 1) / gridDim.x;
    const int64_t kbeg = (int64_t)blockIdx.x * per;
    const int64_t kend = kbeg + per < a.n_pairs ? kbeg + per : a.n_pairs;
    for (int64_t k = kbeg; k < kend && !failed; ++k) {
        const PairRef pr = pair_ref<true>(a.src, k);
        const float *x = (const float *)a.src.A + pr.a_row0 * d;
        const float *y = (const float *)a.src.B + pr.b_row0 * d;
        const int nx = (int)pr.la - 1, ny = (int)pr.lb - 1;
        // slots no chunk writes: pair 0's slot 0 before its own cells, and the
        // last pair's tail slot after its tail
        if (k == 0 || k == a.n_pairs - 1) {
            for (int v = tid; v < 32 * SLOT; v += BT5_T) {
                const int l = v / SLOT, e = v - l * SLOT, w = e / NG, gp = e - w * NG;
                const int g = (gp & 1) ? gp / 2 + NG / 2 : gp / 2;   // inverse of band_gpos
                if (k == 0 && w < g) a.band[band_row(0, l, NG, a.n_pairs * TperR + 1) + band_off(e)] = 0.f;
                if (k == a.n_pairs - 1 && w >= g) a.band[band_row((k + 1) * TperR, l, NG, a.n_pairs * TperR + 1) + band_off(e)] = 0.f;
            }
        }
        for (int P0 = 0; P0 < NPP && !failed; P0 += BT5_M) {
            float4 nb[8];
            __syncthreads();
            {
                // the tile's row increments (padded rows P: real row P - vrows), once
                const int p = P0 + row - a.vrows;
                float4 av[8];
                const bool ok = P0 + row < NPP && p >= 0 && p < nx;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int k4 = half * (K / 8) + i;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (ok && i < K / 8 && k4 < D4) {
                        const float *r0 = x + (int64_t)p * d + 4 * k4, *r1 = r0 + d;
                        const int c = 4 * k4;
                        v.x = c < d ? r1[0] - r0[0] : 0.f;
                        v.y = c + 1 < d ? r1[1] - r0[1] : 0.f;
                        v.z = c + 2 < d ? r1[2] - r0[2] : 0.f;
                        v.w = c + 3 < d ? r1[3] - r0[3] : 0.f;
                    }
                    av[i] = v;
                }
                tc5::store_half(ah, al, row, half, K, av, a.scale);
            }
            auto fetch_cols = [&](int Q0) {
                const int q = Q0 + row - a.NQV;
                const bool ok = Q0 < NQ && Q0 + row < NQ && q >= 0 && q < ny;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int k4 = half * (K / 8) + i;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (ok && i < K / 8 && k4 < D4) {
                        const float *r0 = y + (int64_t)q * d + 4 * k4, *r1 = r0 + d;
                        const int c = 4 * k4;
                        v.x = c < d ? r1[0] - r0[0] : 0.f;
                        v.y = c + 1 < d ? r1[1] - r0[1] : 0.f;
                        v.z = c + 2 < d ? r1[2] - r0[2] : 0.f;
                        v.w = c + 3 < d ? r1[3] - r0[3] : 0.f;
                    }
                    nb[i] = v;
                }
            };
            fetch_cols(0);
            for (int Q0 = 0; Q0 < NQ; Q0 += BT5_N) {
                tc5::store_half(bh, bl, row, half, K, nb, 1.f);
                tc5::fence_async_smem();
                __syncthreads();
                if (tid == 0) {
                    tc5::fence_after();
                    tc5::gemm_split(tmem, ah, al, bh, bl, K, idesc, false);
                    tc5::commit(&mbar);
                }
                fetch_cols(Q0 + BT5_N);
                const bool ok = tc5::mbar_wait(&mbar, phase, max_wait);
                if (__syncthreads_or(!ok)) {
                    failed = true;
                    if (tid == 0) atomicExch(status, (int)SIGK_ETIMEOUT);
                    break;
                }
                phase ^= 1;
                tc5::fence_after();
                {
                    const int r = (warp & 3) * 32 + lane, cb = (warp >> 2) * 64;
#pragma unroll
                    for (int c0 = 0; c0 < 64; c0 += 32) {
                        float v[32];
                        tc5::ld32(tmem + ((unsigned)((warp & 3) * 32) << 16) + (unsigned)(cb + c0), v);
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            *reinterpret_cast<float4 *>(&St[r * BT5_SS + cb + c0 + j]) =
                                make_float4(scheme_coef(v[j], a.src.scheme), scheme_coef(v[j + 1], a.src.scheme),
                                            scheme_coef(v[j + 2], a.src.scheme), scheme_coef(v[j + 3], a.src.scheme));
                    }
                }
                tc5::fence_before();
                __syncthreads();
                // slots with entries in this chunk: pos in [ceil((Q0 - NG + 1) / NG), (Q0 + 127 + NG - 1) / NG]
                const int pos_lo = Q0 / NG, pos_hi = min((Q0 + BT5_N - 1 + NG - 1) / NG, TperR);
                const int l_lo = P0 / NG, l_hi = min(P0 + BT5_M, NPP) / NG;   // lane blocks of this tile
                const int npos4 = (pos_hi - pos_lo + SPW) / SPW;
                const int s = lane / NG, g = lane - s * NG;
                const int gp = band_gpos<NG>(g);
                for (int t = warp; t < (l_hi - l_lo) * npos4; t += BT5_T / 32) {
                    const int l = l_lo + t / npos4;
                    const int pos = pos_lo + (t - (t / npos4) * npos4) * SPW + s;
                    if (pos > pos_hi) continue;
                    const int P = l * NG + g;
                    const float *srow = St + (P - P0) * BT5_SS;
                    // destination slot: the pair's own, or (the tail) the next pair's slot 0
                    const bool tail = pos == TperR;
                    float *dst = a.band + band_row(tail ? (k + 1) * TperR : k * TperR + pos, l, NG, a.n_pairs * TperR + 1);
#pragma unroll
                    for (int w = 0; w < NG; ++w) {
                        const int Q = pos * NG + w - g;
                        const bool own = tail ? (w < g) : (Q >= 0);
                        if (own && Q >= Q0 && Q < Q0 + BT5_N) dst[band_off(w * NG + gp)] = srow[Q - Q0];
                    }
                }
                __syncthreads();
            }
        }
    }
    if (failed) tc5::mbar_wait(&mbar, phase, max_wait);
    tc5::fence_before();
    __syncthreads();
    if (warp == 0) tc5::dealloc(tmem, BT5_N);
}

template <int NG>
cudaError_t launch_coef_tc5(const BandCoefArgs &a, int sms, int *status, cudaStream_t st) {
    const int smem = bt5_smem_bytes(a.src.d);
    auto kern = band_coef_tc5_kernel<NG>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT);
    if (e != cudaSuccess) return e;
    int64_t grid = sms;
    if (grid > a.n_pairs) grid = a.n_pairs;
    kern<<<(int)grid, BT5_T, smem, st>>>(a, status, 1LL << 26);
    return cudaGetLastError();
}

// (R, lambda) with R / 2^lambda in {2, 4, 8}; MINB as fwd_chain.cu
#define SIGK_BAND_CASES(X) \
    X(4, 0, 6) X(4, 1, 6) X(8, 0, 6) X(8, 1, 6) X(8, 2, 6) X(16, 1, 6) X(16, 2, 6) X(16, 3, 6)

bool band_has_instance(int R, int lam) {
#define X(r, l, mb) if (R == r && lam == l) return true;
    SIGK_BAND_CASES(X)
#undef X
    return false;
}

template <int R, int LAM, int MINB>
int band_occupancy() {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, chain_band_kernel<R, LAM, MINB, false>,
                                                      BAND_WARPS * 32, 0) != cudaSuccess)
        return 0;
    return nb;
}

int band_occupancy_of(int R, int lam) {
#define X(r, l, mb) if (R == r && lam == l) return band_occupancy<r, l, mb>();
    SIGK_BAND_CASES(X)
#undef X
    return 0;
}

// ---- the adjoint: the band sweep run backwards in time ----------------------
// The reverse mode of the difference form (as in the strip adjoint of
// fwd_strip.cu): with A(a,b) = dk/dQ(a,b) and V(a,b) = P(a,b) + c(a,b) A(a,b),
//   P(a,b) = c(a,b+1) A(a,b+1) + V(a+1,b),   A(a,b) = A(a,b+1) + P(a,b),
// A(., Nj+1) = 0, V(Ni+1, b) = [b = Nj] g (g the incoming gradient), and
// dk/dc(a,b) = A(a,b) (K(a,b-1) + K(a-1,b)).  Running the chain's schedule
// backwards (rows ascending within a step) has every input ready, as in the
// strip adjoint.  The sums K(a,b-1) + K(a-1,b) are not stored: the forward
// step is undone in place,
//   K(a,b-1) = K(a,b) - Q(a,b),   Q(a-1,b) = Q(a,b) - c(a,b) (K(a,b-1) + K(a-1,b)),
// from the state after the step, exact up to rounding, with the state reset
// to the forward's own every BAND_CK macro-steps (checkpoints), the K a row
// had when it left its pair (exit states: the forward resets K to 1 there),
// and the last row's Q before each step (it has no row below to recover it
// from).  dk/dc is summed per coarse cell in registers and stored densely.

struct BandAdjArgs {
    PairSrc src;            // oriented: rows refine the A paths
    const float *band;      // coefficients, band layout
    const float *ckpt, *exitk, *botq;
    int nck;
    int64_t bq_stride;
    const float *gout;      // incoming gradient, indexed like the forward's outputs
    float *gband;           // dk/dc (unscaled) in the band layout, TperR + 1 slots per pair
                            // (slot TperR: the pair's tail), unpacked by band_gbar_kernel
    int64_t n_pairs, ppw;
    int TperR, NQ, NQV, vrows, nx, ny;
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// dk/dc from the adjoint's band layout into the dense Gbar the chain-rule
// contractions read: [row path * nx][column path * ny] (Gram: every column
// path of the call; pairs: one nx x ny block per pair).  Pair k's cell (P, Q)
// = (l NG + g, Q) is in slot (k, pos) window w with pos NG + w = Q + g (slot
// TperR: the tail).  A block takes gb_pos(NG) positions of one pair: it
// stages those slots and the next one in shared memory (coalesced), then
// writes the real cells of columns Q in [pos0 NG, (pos0 + gb_pos) NG) row by
// row, each row a contiguous run (window rows staged NG + 1 floats apart):
// 32 columns (128 bytes) a row for NG <= 4, 32 for NG = 8 (four positions,
// the static shared memory's limit).
__host__ __device__ constexpr int gb_pos(int NG) { return NG <= 4 ? 8 : 4; }
constexpr int GB_THREADS = 256;
// position groups per pair: the columns Q < NQ = TperR NG, and for the
// surface also Q = NQ (its last node column, in the tail slot)
__host__ __device__ inline int gb_groups(int TperR, bool surf, int NG) {
    return (TperR + (surf ? 1 : 0) + gb_pos(NG) - 1) / gb_pos(NG);
}

struct BandGbarArgs {
    PairSrc src;
    const float *gband;
    float *gbar;
    int64_t g_ld;           // floats per gbar row
    int64_t a_first;        // first A path of this launch (rows of gbar count from it)
    int gram;               // 1: gbar columns hold every B path of the call
    int64_t n_pairs;
    int TperR, NQV, vrows, nx, ny;
    // surface mode (s_pair > 0): the band holds the sweep's values at the
    // sample-grid nodes, node (p + 1, q + q_off) of cell (p, q) (q_off = 1 at
    // dyadic order 0, where the stored node is the cell's lower-right corner;
    // 0 above, the lower-left one, the last column coming from the tail slot);
    // they go to gbar[(kbase + k) s_pair + (p + 1) s_a + (q + q_off) s_b]
    int64_t s_pair, s_a, s_b;
    int q_off;
};

template <int NG>
__global__ void __launch_bounds__(GB_THREADS) band_gbar_kernel(BandGbarArgs a) {
    constexpr int SLOT = NG * NG;
    constexpr int NP = 32 * NG;                 // padded rows
    constexpr int GB_POS = gb_pos(NG);
    constexpr int SPAN = GB_POS * NG;           // columns per block task
    constexpr int WS = NG + 1;                  // staged window row stride: consecutive
                                                // columns of a row hit distinct banks
    constexpr int SS = NG * WS;                 // staged slot stride
    __shared__ float sl[(GB_POS + 1) * 32 * SS];
    const int ngroups = gb_groups(a.TperR, a.s_pair > 0, NG);
    const int64_t tasks = a.n_pairs * ngroups;
    for (int64_t t = blockIdx.x; t < tasks; t += gridDim.x) {
        const int64_t k = t / ngroups;
        const int pos0 = (int)(t - k * ngroups) * GB_POS;
        const int npos = min(GB_POS + 1, a.TperR + 1 - pos0);   // slots pos0 .. pos0 + npos - 1
        __syncthreads();
        const float4 *src = reinterpret_cast<const float4 *>(a.gband + ((k * (a.TperR + 1) + pos0) * 32) * (int64_t)SLOT);
        for (int v = threadIdx.x; v < npos * 32 * SLOT / 4; v += GB_THREADS) {
            const float4 x = src[v];
            const int slot = v / (SLOT / 4), e = (v - slot * (SLOT / 4)) * 4;
            float *d = sl + slot * SS;
            d[(e / NG) * WS + e % NG] = x.x;
            d[((e + 1) / NG) * WS + (e + 1) % NG] = x.y;
            d[((e + 2) / NG) * WS + (e + 2) % NG] = x.z;
            d[((e + 3) / NG) * WS + (e + 3) % NG] = x.w;
        }
        __syncthreads();
        const bool surf = a.s_pair > 0;
        float *base;
        int64_t sr = a.g_ld, sc = 1;
        if (surf) {
            base = a.gbar + (a.src.kbase + k) * a.s_pair + a.s_a;   // node row p + 1
            sr = a.s_a;
            sc = a.s_b;
        } else {
            const PairRef pr = pair_ref<true>(a.src, k);
            const int64_t ia = pr.a_row0 / a.src.La - a.a_first;
            const int64_t jb = a.gram ? pr.b_row0 / a.src.Lb : 0;
            base = a.gbar + ia * a.nx * a.g_ld + jb * a.ny;
        }
        // surface: column 0 too when the pairs have virtual columns at the
        // left (NQV >= 1 at dyadic orders >= 1): there the stored node is the
        // boundary value, exactly 1 (c = 0 keeps K = 1 and Q = 0), and the
        // border fill need not write that strided column; without them the
        // slot holds the previous pair's last column instead
        const int qlo = surf && a.q_off == 0 && a.NQV == 0 ? 1 : 0;
        const int qhi = surf ? a.ny - a.q_off : a.ny - 1;
        if (surf) base += (int64_t)a.q_off * sc;
        const int Qlo = pos0 * NG;
        for (int v = threadIdx.x; v < NP * SPAN; v += GB_THREADS) {
            const int P = v / SPAN, Q = Qlo + (v - (v / SPAN) * SPAN);
            const int p = P - a.vrows, q = Q - a.NQV;
            if (p < 0 || p >= a.nx || q < qlo || q > qhi) continue;
            const int l = P / NG, g = P - (P / NG) * NG;
            const int tq = Q + g, pos = tq / NG, w = tq - (tq / NG) * NG;   // pos - pos0 in [0, npos)
            base[(int64_t)p * sr + (int64_t)q * sc] = sl[((pos - pos0) * 32 + l) * SS + w * WS + band_gpos<NG>(g)];
        }
    }
}

// macro-steps of coefficient slots and last-row Q's kept per warp
template <int R, int LAM>
__host__ __device__ constexpr int adj_ring() {
    constexpr int d = band_ring<R, (R >> LAM)>();
    return d > 0 ? d : 2;
}
template <int R, int LAM>
__host__ __device__ constexpr int adj_warp_floats() {
    return adj_ring<R, LAM>() * (32 * (R >> LAM) * (R >> LAM) + R);
}

template <int R, int LAM>
__global__ void __launch_bounds__(BAND_WARPS * 32, 6) chain_band_adj_kernel(BandAdjArgs a) {
    constexpr int S = 1 << LAM;
    constexpr int NG = R / S;
    constexpr int H = R / 2;
    constexpr int NH = NG / 2;
    constexpr int JOUT = R - 2;
    constexpr int SLOT = NG * NG;
    constexpr int NCH = SLOT >= 4 ? SLOT / 4 : 1;   // 16-byte chunks of a lane's slot
    extern __shared__ __align__(16) float adj_sm[];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int64_t gw = (int64_t)blockIdx.x * BAND_WARPS + warp;
    const int64_t k0 = gw * a.ppw;
    if (k0 >= a.n_pairs) return;
    const int np = (int)min(a.ppw, a.n_pairs - k0);
    const int TperR = a.TperR;
    // per warp: D macro-steps of coefficient slots (lane-major, 16-byte
    // chunks rotated by lane against bank conflicts) and of the last row's Q
    constexpr bool DEEP = band_ring<R, NG>() > 0;   // fetched D - 1 macro-steps ahead, else one
    constexpr int D = adj_ring<R, LAM>();
    float *ring = adj_sm + (size_t)warp * adj_warp_floats<R, LAM>();
    float *bqs = ring + D * 32 * SLOT;
    const float *bq = a.botq + gw * a.bq_stride;
    auto chunk = [&](int c) { return NCH >= 8 ? (c ^ (lane & 7)) : (NCH >= 2 ? (c ^ (lane & (NCH - 1))) : c); };
    auto lane_slot = [&](int buf) { return ring + ((size_t)buf * 32 + lane) * SLOT; };

    auto locate = [&](int64_t m, int &kl, int &pos) {
        const int64_t mm = m - lane;
        int64_t q = mm >= 0 ? mm / TperR : -((-mm + TperR - 1) / TperR);
        kl = (int)q;
        pos = (int)(mm - q * TperR);
    };
    // the lane's slot in macro-step m, as in the forward
    const int64_t nslots = a.n_pairs * TperR + 1;
    auto slot_ptr = [&](int64_t m) -> const float * {
        return m >= lane && m - lane <= (int64_t)np * TperR
                   ? a.band + band_row(k0 * TperR + m - lane, lane, NG, nslots) : nullptr;
    };
    // window w of macro-step m (slot src, null outside the chain) into buffer m % D;
    // with window NG-1 also the last row's Q
    auto fetch = [&](int64_t m, const float *src, int w) {
        float *dst = lane_slot((int)(m % D));
        if constexpr (NG == 8) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float *dd = dst + 4 * chunk(2 * w + h);
                if (src) cp_async<16>(dd, src + band_off(w * NG + 4 * h));
                else *reinterpret_cast<float4 *>(dd) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        } else if constexpr (NG == 4) {
            float *dd = dst + 4 * chunk(w);
            if (src) cp_async<16>(dd, src + band_off(w * NG));
            else *reinterpret_cast<float4 *>(dd) = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            float *dd = dst + 2 * w;
            if (src) cp_async<8>(dd, src + band_off(w * NG));
            else *reinterpret_cast<float2 *>(dd) = make_float2(0.f, 0.f);
        }
        if (w == NG - 1 && lane == 31) {
            float *bd = bqs + (m % D) * R;
#pragma unroll
            for (int h = 0; h < R / 4; ++h) cp_async<16>(bd + 4 * h, bq + m * R + 4 * h);
        }
    };
    auto read_window = [&](int buf, int w, float2 (&c)[NH]) {
        const float *sl = lane_slot(buf);
        float v[NG];
        if constexpr (NG == 8) {
            const float4 x0 = *reinterpret_cast<const float4 *>(sl + 4 * chunk(2 * w));
            const float4 x1 = *reinterpret_cast<const float4 *>(sl + 4 * chunk(2 * w + 1));
            v[0] = x0.x; v[1] = x0.y; v[2] = x0.z; v[3] = x0.w;
            v[4] = x1.x; v[5] = x1.y; v[6] = x1.z; v[7] = x1.w;
        } else if constexpr (NG == 4) {
            const float4 x0 = *reinterpret_cast<const float4 *>(sl + 4 * chunk(w));
            v[0] = x0.x; v[1] = x0.y; v[2] = x0.z; v[3] = x0.w;
        } else {
            const float2 x0 = *reinterpret_cast<const float2 *>(sl + 2 * w);
            v[0] = x0.x; v[1] = x0.y;
        }
#pragma unroll
        for (int g = 0; g < NH; ++g) c[g] = make_float2(v[2 * g], v[2 * g + 1]);   // groups g, g + NH
    };

    // forward state as (K, -Q): undoing a step then needs no negation
    float2 KP[H], QN[H], A[H], V[H];
    float2 gN[NH], gO[NH];
    // coefficients of the window processed before (the next one in forward
    // order): a row's coefficient one forward step later comes from these or
    // from the current window's
    float2 CNP[NH];
#pragma unroll
    for (int i = 0; i < H; ++i) {
        A[i] = make_float2(0.f, 0.f); V[i] = A[i];
        KP[i] = make_float2(1.f, 1.f); QN[i] = A[i];
    }
#pragma unroll
    for (int g = 0; g < NH; ++g) { gN[g] = make_float2(0.f, 0.f); gO[g] = gN[g]; CNP[g] = gN[g]; }

    const int64_t mlast = (int64_t)np * TperR + 31;
    int kl, pos;   // this lane's pair and position at macro-step m, tracked backwards
    locate(mlast, kl, pos);
    if constexpr (DEEP) {
#pragma unroll 1
        for (int64_t m = mlast; m > mlast - (D - 1); --m) {
            if (m >= 0) {
                const float *s0 = slot_ptr(m);
#pragma unroll
                for (int w = NG - 1; w >= 0; --w) fetch(m, s0, w);
            }
            cp_commit();
        }
    } else {
        const float *s0 = slot_ptr(mlast);
#pragma unroll
        for (int w = NG - 1; w >= 0; --w) {
            fetch(mlast, s0, w);
            cp_commit();
        }
    }

    for (int64_t m = mlast; m >= 0; --m) {
        if (m != mlast && --pos < 0) {
            pos = TperR - 1;
            --kl;
        }
        const bool trans = (pos == 0);
        const float *sprev = nullptr;
        if constexpr (DEEP) {
            if (m >= D - 1) {
                const float *s0 = slot_ptr(m - (D - 1));
#pragma unroll
                for (int w = NG - 1; w >= 0; --w) fetch(m - (D - 1), s0, w);
            }
            cp_commit();
            cp_wait<D - 2>();   // macro-steps m and m - 1
        } else if (m >= 1) {
            sprev = slot_ptr(m - 1);
        }
        // what macro-step m - 1 will read from memory: a checkpoint, its exit states
        // (the forward wrote them to DRAM long ago: about 1 GB for 16384 pairs)
        if (m % BAND_CK == 0 && m >= 1)
            prefetch_l2(a.ckpt + ((gw * a.nck + (m - 1) / BAND_CK) * 32 + lane) * (int64_t)(2 * R));
        if (pos == 1 && kl >= 1 && kl <= np) prefetch_l2(a.exitk + ((k0 + kl - 1) * 32 + lane) * (int64_t)R);
        if ((m + 1) % BAND_CK == 0 || m == mlast) {
            // the forward's state after macro-step m
            const float4 *ck = reinterpret_cast<const float4 *>(
                a.ckpt + ((gw * a.nck + m / BAND_CK) * 32 + lane) * (int64_t)(2 * R));
#pragma unroll
            for (int i = 0; i < H; i += 2) {
                const float4 kk4 = ck[i / 2], qq4 = ck[H / 2 + i / 2];
                KP[i] = make_float2(kk4.x, kk4.y); KP[i + 1] = make_float2(kk4.z, kk4.w);
                QN[i] = make_float2(-qq4.x, -qq4.y); QN[i + 1] = make_float2(-qq4.z, -qq4.w);
            }
        }
        const bool cur_ok = kl >= 0 && kl < np, prev_ok = kl >= 1 && kl <= np;
        // the lane's slot rows in the dk/dc band: this pair's position, and at
        // position 0 also the previous pair's tail slot (its cells with w < g)
        float *gs_cur = cur_ok ? a.gband + (((k0 + kl) * (TperR + 1) + pos) * 32 + lane) * (int64_t)SLOT : nullptr;
        float *gs_prev = (trans && prev_ok)
                             ? a.gband + (((k0 + kl - 1) * (TperR + 1) + TperR) * 32 + lane) * (int64_t)SLOT
                             : nullptr;
        // rows turning over in this macro-step leave pair kl - 1 in reverse;
        // lane 31 seeds that pair's incoming gradient at its corner
        float gseed = 0.f;
        const bool has_prev = trans && prev_ok;
        float exK[R];   // their K when they left it (rows 0 .. R-1)
#pragma unroll
        for (int i = 0; i < R; ++i) exK[i] = 1.f;
        if (has_prev) {
            const float4 *ex = reinterpret_cast<const float4 *>(a.exitk + ((k0 + kl - 1) * 32 + lane) * (int64_t)R);
#pragma unroll
            for (int i = 0; i < R / 4; ++i) {
                const float4 v = ex[i];
                exK[4 * i] = v.x; exK[4 * i + 1] = v.y; exK[4 * i + 2] = v.z; exK[4 * i + 3] = v.w;
            }
            if (lane == 31) {
                // a symmetric Gram's pair (i, j), i < j, stands for (j, i) too
                const PairRef pr = pair_ref<true>(a.src, k0 + kl - 1);
                gseed = a.gout[pr.out0] + (pr.out1 >= 0 ? a.gout[pr.out1] : 0.f);
            }
        }
        const int buf = (int)(m % D), bufn = (int)((m + D - 1) % D);   // bufn: macro-step m - 1's

        // a runtime loop over the windows keeps the body within the instruction cache
#pragma unroll 1
        for (int w = NG - 1; w >= 0; --w) {
            if constexpr (!DEEP) {
                if (m >= 1) fetch(m - 1, sprev, w);
                cp_commit();
                cp_wait<NG - 1>();   // window w - 1 of this macro-step (w = 0: window NG-1 of the one before)
            }
            float2 CN[NH], CO[NH];
            read_window(buf, w, CN);
            if (w > 0) read_window(buf, w - 1, CO);
            else read_window(bufn, NG - 1, CO);
            const int tw = has_prev ? w : -1;   // group whose rows turn over in this window

#pragma unroll
            for (int jj = S - 1; jj >= 0; --jj) {
                const int j = w * S + jj;
                const float qbot = bqs[buf * R + j];          // lane 31: its last row's Q before the step
                const float vH = V[0].y;
                float vd = __shfl_down_sync(FULL, V[0].x, 1);
                if (lane == 31) vd = (has_prev && j == JOUT) ? gseed : 0.f;
                // packed rows (H-1, R-1) first: their K before the step is the
                // row above packed row 0's
                constexpr int gH = (H - 1) / S, sH = (H - 1) % S;
                const bool hx = jj == sH && tw == gH, hy = jj == sH && tw == gH + NH;
                float2 KlH = add2(KP[H - 1], QN[H - 1]);
                float2 KpH = make_float2(hx ? exK[H - 1] : KlH.x, hy ? exK[R - 1] : KlH.y);
                KlH = make_float2(hx ? 1.f : KlH.x, hy ? 1.f : KlH.y);
                float pKs = __shfl_up_sync(FULL, KpH.y, 1);
                if (lane == 0) pKs = 1.f;
                float2 kprev = make_float2(pKs, KpH.x);
                float2 t0 = make_float2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    const int g1 = i / S, s1 = i % S;
                    const bool px = jj == s1 && tw == g1, py = jj == s1 && tw == g1 + NH;
                    float2 Kl, Kp;
                    if (i == H - 1) {
                        Kl = KlH;
                        Kp = KpH;
                    } else {
                        Kl = add2(KP[i], QN[i]);
                        Kp = Kl;
                        if (jj == s1) {
                            Kp = make_float2(px ? exK[i] : Kl.x, py ? exK[i + H] : Kl.y);
                            Kl = make_float2(px ? 1.f : Kl.x, py ? 1.f : Kl.y);
                        }
                    }
                    const float2 sum = add2(Kl, kprev);
                    const float2 c = (jj >= s1) ? CN[g1] : CO[g1];
                    const float2 tq = fma2(c, sum, QN[i]);   // -Q before the step of the rows above
                    if (i == 0) t0 = tq;
                    else QN[i - 1] = tq;
                    KP[i] = Kp;
                    kprev = Kp;
                    const float2 vb = (i < H - 1) ? V[i < H - 1 ? i + 1 : 0] : make_float2(vH, vd);
                    // the row's coefficient one forward step later
                    const float2 cp = (jj < S - 1) ? ((jj + 1 >= s1) ? CN[g1] : CO[g1])
                                                   : (s1 == 0 ? CNP[g1] : CN[g1]);
                    const float2 P = fma2(cp, A[i], vb);
                    float2 An = add2(A[i], P);
                    V[i] = fma2(c, An, P);
                    if (jj >= s1) gN[g1] = fma2(An, sum, gN[g1]);
                    else gO[g1] = fma2(An, sum, gO[g1]);
                    // in reverse the row enters its previous pair: A(., Nj+1) = 0
                    if (jj == s1) An = make_float2(px ? 0.f : An.x, py ? 0.f : An.y);
                    A[i] = An;
                }
                float qd = __shfl_down_sync(FULL, t0.x, 1);
                if (lane == 31) qd = -qbot;
                QN[H - 1] = make_float2(t0.y, qd);
            }
            // window w's cells are complete: (P, Q) = (lane*NG + g, pos*NG + w - g),
            // in the order of the band's groups (g, g + NH side by side): one
            // vector store of the window row per slot
            if (a.src.scheme != SIGK_SCHEME_EXPLICIT) {   // dk/dc' -> dk/dc of the cell's coefficient
#pragma unroll
                for (int g = 0; g < NH; ++g) {
                    gN[g].x *= scheme_dcoef(CN[g].x, a.src.scheme);
                    gN[g].y *= scheme_dcoef(CN[g].y, a.src.scheme);
                }
            }
            if (gs_cur) store_window<NG>(gs_cur + w * NG, gN);
            if (gs_prev) store_window<NG>(gs_prev + w * NG, gN);
#pragma unroll
            for (int g = 0; g < NH; ++g) { gN[g] = gO[g]; gO[g] = make_float2(0.f, 0.f); CNP[g] = CN[g]; }
        }
    }
    cp_wait<0>();
}

// Real (unpadded) increments of paths: inc[(path * (L - 1) + p) * d + c], of the
// row role's and the column role's paths in one launch (a small gradient step
// is bound by its launches), which also clears the status word of the
// workspace (null: left alone).
struct IncJob {
    const float *pts;
    int64_t npaths, L;
    float *inc;
};
__global__ void band_inc_kernel(IncJob ja, IncJob jb, int64_t d, int *status) {
    if (status && blockIdx.x == 0 && threadIdx.x == 0) *status = 0;
    const int64_t na = ja.npaths * (ja.L - 1) * d, total = na + jb.npaths * (jb.L - 1) * d;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < total;
         u += (int64_t)gridDim.x * blockDim.x) {
        const bool isb = u >= na;
        const IncJob &j = isb ? jb : ja;
        const int64_t v = isb ? u - na : u, c = v % d, row = v / d;
        const int64_t path = row / (j.L - 1), p = row - path * (j.L - 1);
        const float *x = j.pts + (path * j.L + p) * d + c;
        j.inc[v] = x[d] - x[0];
    }
}

// The chain rule through G(p, q) = <dx_p, dy_q>: C (+)= G B per batch, where
// G is dk/dc read straight from the adjoint's band layout (pair k's value at
// row-role increment p, column-role increment q sits in slot (k, pos, lane)
// at [w][gpos(g)] with P = p + vrows = lane NG + g, Q = q + NQV = pos NG + w - g).
// Not trans: C rows are the row role's increments (all row paths), the sum
// runs over the column role's; trans: the other way round.  Output tiles are
// 128 band coordinates (P, or Q when trans) of one output path by 32
// channels; reduction slices are 32 band coordinates of one reduction path.
// A slice's slots are staged whole (contiguous 16-byte loads), then
// transposed into the tile in shared memory; virtual rows and columns (the
// band's padding) read as zero.  4 x 4 outputs per thread; long reductions
// are split across blocks whose partial tiles a second kernel sums in order.
struct GemmArgs {
    const float *G;          // dense dk/dc (the tensor-core contraction only)
    int64_t g_ld;
    const float *Bm;
    int64_t b_bstride;
    float *C;
    int64_t c_bstride;
    int64_t M, K;            // output rows, reduction length (real increments)
    int N, trans, ksplit;    // ksplit > 1 (one batch only): block ks writes its partial
    float *partial;          // tile to partial[ks][M][N], summed by band_split_sum_kernel
    int64_t tri_rb, tri_cb;  // symmetric Gram: only pairs i <= j are stored (tensor-core path)
    const float *band;
    int mode;                // PM_PAIRS: batch b is pair b; PM_GRAM / PM_GRAM_SYM: one batch
    int64_t nb, a0, kbase;   // Gram: column paths, the launch's first row path, its first pair
    int64_t nA, nB;          // row / column paths of a batch (1 and 1 for pairs)
    int TperR1, vrows, NQV, nx, ny;
};
constexpr int GEMM_MAX_SPLIT = 8;
constexpr int GT_M = 128, GT_K = 32, GT_N = 32;

// the launch-local pair of row path ia and column path jb (-1: none stored,
// below a symmetric Gram's diagonal)
__device__ __forceinline__ int64_t gemm_pair(const GemmArgs &a, int64_t b, int64_t ia, int64_t jb) {
    if (a.mode == PM_PAIRS) return b;
    if (a.mode == PM_GRAM) return (a.a0 + ia) * a.nb + jb - a.kbase;
    if (ia > jb) return -1;
    return ia * a.nb - ia * (ia - 1) / 2 + (jb - ia) - a.kbase;
}

template <int NG>
__global__ void __launch_bounds__(256) band_gemm_kernel(GemmArgs a) {
    constexpr int SLOT = NG * NG;
    constexpr int BH = 32 * NG;                                           // band rows of a path
    constexpr int TL0 = (BH < GT_M ? BH : GT_M) / NG, TP0 = GT_K / NG + 1;   // staged lanes, positions
    constexpr int TL1 = GT_K / NG, TP1 = GT_M / NG + 1;                      // (trans)
    constexpr int ST0 = TL0 * TP0 * SLOT, ST1 = TL1 * TP1 * SLOT;
    constexpr int STF = ST0 > ST1 ? ST0 : ST1;
    constexpr int SV = (STF / 4 + 255) / 256;   // staged float4s per thread
    __shared__ __align__(16) float Gs[GT_K][GT_M + 4];
    __shared__ __align__(16) float Bs[GT_K][GT_N];
    __shared__ __align__(16) float St[STF];
    const bool tr = a.trans != 0;
    const int64_t b = blockIdx.z / a.ksplit;
    const int ks = blockIdx.z - (int)b * a.ksplit;
    const float *Bm = a.Bm + b * a.b_bstride;
    float *C = a.C + b * a.c_bstride;
    const int NQ = (a.TperR1 - 1) * NG;   // band columns of a path
    const int ocoords = tr ? NQ : BH;     // output band coordinates of a path
    const int tpp = (ocoords + GT_M - 1) / GT_M;
    const int64_t opath = blockIdx.x / tpp;
    const int o0 = (int)(blockIdx.x - opath * tpp) * GT_M;
    const int n0 = blockIdx.y * GT_N;
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
    // the reduction: paths [rlo, rhi) (a symmetric Gram stores pairs i <= j
    // only), each in spp slices of 32 band coordinates
    const int rcoords = tr ? BH : NQ;
    const int spp = (rcoords + GT_K - 1) / GT_K;
    int64_t rlo = 0, rhi = tr ? a.nA : a.nB;
    if (a.mode == PM_GRAM_SYM) {
        if (tr) rhi = opath + 1; else rlo = opath;
    }
    const int64_t total = (rhi - rlo) * spp;
    const int64_t s_lo = total * ks / a.ksplit, s_hi = total * (ks + 1) / a.ksplit;
    const int TL = tr ? TL1 : TL0, TP = tr ? TP1 : TP0;
    const int SN = TL * TP * SLOT / 4;   // float4s staged a slice
    const int nrr = tr ? a.nx : a.ny;    // real increments of the reduction role
    const int nro = tr ? a.ny : a.nx;    // and of the output role
    const int vro = tr ? a.NQV : a.vrows, vrr = tr ? a.vrows : a.NQV;

    float4 sv[SV];
    float br[4];
    int c0n = 0;
    // slice sidx into registers: its slots (not trans: lanes o0/NG + [0, TL0),
    // positions c0/NG + [0, TP0); trans: lanes c0/NG + [0, TL1), positions
    // o0/NG + [0, TP1); positions past the pair's last slot read as zero) and
    // the reduction role's 32 increments of 32 channels
    auto load = [&](int64_t sidx) {
        const int64_t rp = rlo + sidx / spp;
        const int c0 = (int)(sidx - (rp - rlo) * spp) * GT_K;
        const int64_t k = tr ? gemm_pair(a, b, rp, opath) : gemm_pair(a, b, opath, rp);
        const int l0 = (tr ? c0 : o0) / NG, p0 = (tr ? o0 : c0) / NG;
#pragma unroll
        for (int i = 0; i < SV; ++i) {
            const int u = threadIdx.x + 256 * i;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (u < SN && k >= 0) {
                const int sl = u / (SLOT / 4), e = u - sl * (SLOT / 4);
                const int pr = sl / TL, lr = sl - pr * TL;
                const int pos = p0 + pr;
                if (pos < a.TperR1)
                    v = __ldg(reinterpret_cast<const float4 *>(
                                  a.band + ((k * a.TperR1 + pos) * 32 + l0 + lr) * (int64_t)SLOT) + e);
            }
            sv[i] = v;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int v = threadIdx.x + 256 * i;
            const int kk = v / GT_N, nn = v % GT_N;
            const int real = c0 + kk - vrr;
            const int n = n0 + nn;
            br[i] = (real >= 0 && real < nrr && n < a.N && k >= 0) ? Bm[(rp * nrr + real) * a.N + n] : 0.f;
        }
        c0n = c0;
    };
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int jx = 0; jx < 4; ++jx) acc[i][jx] = 0.f;
    if (s_lo < s_hi) load(s_lo);
    for (int64_t sidx = s_lo; sidx < s_hi; ++sidx) {
        const int c0 = c0n;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SV; ++i) {
            const int u = threadIdx.x + 256 * i;
            if (u < SN) reinterpret_cast<float4 *>(St)[u] = sv[i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int v = threadIdx.x + 256 * i;
            Bs[v / GT_N][v % GT_N] = br[i];
        }
        __syncthreads();
        // Gs[kk][rr]: output coordinate o0 + rr, reduction coordinate c0 + kk;
        // virtual rows and columns of the reduction role read as zero
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int v = threadIdx.x + 256 * i;
            const int rr = v % GT_M, kk = v / GT_M;
            const int Prel = tr ? kk : rr, Qrel = tr ? rr : kk;
            const int lr = Prel / NG, g = Prel % NG;
            const int t = Qrel + g, pr = t / NG, w = t % NG;
            const int real = c0 + kk - vrr;
            const bool ok = real >= 0 && real < nrr && (tr || o0 + rr < BH);
            Gs[kk][rr] = ok ? St[(pr * TL + lr) * SLOT + w * NG + band_gpos<NG>(g)] : 0.f;
        }
        if (sidx + 1 < s_hi) load(sidx + 1);
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < GT_K; ++kk) {
            const float4 gv = *reinterpret_cast<const float4 *>(&Gs[kk][4 * ty]);
            const float4 bv = *reinterpret_cast<const float4 *>(&Bs[kk][4 * tx]);
            const float gg[4] = {gv.x, gv.y, gv.z, gv.w};
            const float bb[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int jx = 0; jx < 4; ++jx) acc[i][jx] = fmaf(gg[i], bb[jx], acc[i][jx]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int oc = o0 + 4 * ty + i;
        const int real = oc - vro;
        if (oc >= ocoords || real < 0 || real >= nro) continue;
        const int64_t r = opath * nro + real;
#pragma unroll
        for (int jx = 0; jx < 4; ++jx) {
            const int n = n0 + 4 * tx + jx;
            if (n >= a.N) continue;
            if (a.ksplit > 1) a.partial[((int64_t)ks * a.M + r) * a.N + n] = acc[i][jx];
            else C[r * a.N + n] = acc[i][jx];
        }
    }
}

// The same contraction with the row role's increments as output (not trans), for
// lanes of 4 or 8 coarse rows: no tile is turned.  A thread owns the NG rows of a
// lane and four channels (a block: 128 rows by 32 channels, as above), and takes
// the lane's slots as they lie: window w holds the pairs (dk/dc of row h, of row
// h + NG/2), which meet the columns j = NG - 1 + w - h and j - NG/2 of the
// position; the column increments are kept in shared memory as those pairs, so
// a window is NG/2 float2s of dk/dc, one new pair of column rows and 2 NG packed
// FMAs with no moves, about half of the FP32 pipe's time in shared-memory
// wavefronts.  POS positions (32 columns) a stage, double-buffered: slots by
// cp.async, the columns through registers.  Each output adds the columns of its
// share of the reduction in the same order as band_gemm_kernel, bit for bit (a
// Gram's gradients are sums of 10^4 terms that cancel: another order moves them by
// 1e-5).  128 x 128 Gram of 256-point paths, N = 32: 2.98 ms a launch through
// turned tiles (which still take two rows a lane), 2.3 here.
template <int NG>
struct GrStage {
    static constexpr int LANES = 128 / NG, THREADS = 8 * LANES;
    static constexpr int POS = 32 / NG, SLOT = NG * NG, SS = SLOT + 4;   // padded: 4 lanes, 4 bank quads
    static constexpr int ROWS = (POS + 1) * NG;                          // column rows, from NG - 1 before the stage's first
    float g[POS][LANES][SS];
    float y[ROWS][2][8][4];   // row j: for channel quad c, halves of the pairs (y[j], y[j - NG/2]) of its 4 channels
};

template <int NG>
__global__ void __launch_bounds__(GrStage<NG>::THREADS, 512 / GrStage<NG>::THREADS) band_rows_kernel(GemmArgs a) {
    using St = GrStage<NG>;
    constexpr int NH = NG / 2, POS = St::POS, SLOT = St::SLOT, ROWS = St::ROWS, NT = St::THREADS, LANES = St::LANES;
    constexpr int YV = (ROWS * 32 + NT - 1) / NT;   // column values a thread stages
    extern __shared__ __align__(16) float gr_sm[];
    St *st = reinterpret_cast<St *>(gr_sm);         // two of them
    const int tid = threadIdx.x, l = tid >> 3, cq = tid & 7;
    const int64_t b = blockIdx.z / a.ksplit;
    const int ks = blockIdx.z - (int)b * a.ksplit;
    const float *Bm = a.Bm + b * a.b_bstride;
    float *C = a.C + b * a.c_bstride;
    constexpr int TPP = 32 / LANES;                 // blocks a path
    const int64_t opath = blockIdx.x / TPP;
    const int l0 = (int)(blockIdx.x - opath * TPP) * LANES;
    const int n0 = blockIdx.y * 32;
    // the share in slices of 32 columns; a slice is POS positions, and cells of
    // its last columns lie in the position after it
    const int TperR = a.TperR1 - 1, spp = (TperR + POS - 1) / POS;
    const int64_t rlo = a.mode == PM_GRAM_SYM ? opath : 0;
    const int64_t total = (a.nB - rlo) * spp;
    const int64_t s_lo = total * ks / a.ksplit, s_hi = total * (ks + 1) / a.ksplit;

    // a stage: positions p .. of path rp, which the share visits from pb to pe
    struct Walk { int64_t rp; int p, pb, pe; };
    auto open = [&](int64_t path, int slice) {
        Walk w;
        w.rp = path;
        w.pb = w.p = slice * POS;
        const int64_t left = s_hi - path * spp;   // slices of this path before the share's end
        w.pe = left >= spp ? TperR : (int)left * POS;
        return w;
    };
    auto next = [&](const Walk &w) {
        if (w.p + POS <= w.pe) {
            Walk n = w;
            n.p += POS;
            return n;
        }
        return open(w.rp + 1, 0);
    };
    auto ended = [&](const Walk &w) { return w.rp * spp >= s_hi; };

    float yr[YV];
    // a stage's slots into buffer buf (cp.async), its columns into registers
    auto fetch = [&](const Walk &w, int buf) {
        const int64_t k = gemm_pair(a, b, opath, rlo + w.rp);
        const float *src = a.band + ((k * a.TperR1 + w.p) * 32 + l0) * (int64_t)SLOT;
#pragma unroll
        for (int i = 0; i < POS * LANES * (SLOT / 4) / NT; ++i) {
            const int v = tid + NT * i, sl = v / (SLOT / 4), e = v - sl * (SLOT / 4), pr = sl / LANES, lr = sl % LANES;
            float *dst = &st[buf].g[pr][lr][4 * e];
            if (w.p + pr <= w.pe) cp_async<16>(dst, src + (pr * 32 + lr) * SLOT + 4 * e);
        }
        cp_commit();
#pragma unroll
        for (int i = 0; i < YV; ++i) {
            const int v = tid + NT * i, j = v >> 5, n = n0 + (v & 31);
            const int q = (w.p - 1) * NG + j + 1 - a.NQV;   // row j: Q = p NG - (NG - 1) + j
            yr[i] = j < ROWS && q >= 0 && q < a.ny && n < a.N ? __ldg(Bm + ((rlo + w.rp) * a.ny + q) * a.N + n) : 0.f;
        }
    };
    auto put_y = [&](int buf) {
#pragma unroll
        for (int i = 0; i < YV; ++i) {
            const int v = tid + NT * i, j = v >> 5, c = v & 31;
            if (j >= ROWS) continue;
            // channel c of quad c / 4: pair c % 2 of half (c % 4) / 2
            st[buf].y[j][(c & 3) >> 1][c >> 2][2 * (c & 1)] = yr[i];
            if (j + NH < ROWS) st[buf].y[j + NH][(c & 3) >> 1][c >> 2][2 * (c & 1) + 1] = yr[i];
        }
    };
    float2 acc[NH][4];
#pragma unroll
    for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[h][c] = make_float2(0.f, 0.f);

    Walk wn = open(s_lo / spp, (int)(s_lo % spp));
    if (s_lo < s_hi) fetch(wn, 0);
    for (int buf = 0; s_lo < s_hi && !ended(wn); buf ^= 1) {
        const Walk wk = wn;
        wn = next(wk);
        put_y(buf);
        cp_wait<0>();
        __syncthreads();   // the stage is complete, and the other buffer's readers are done
        if (!ended(wn)) fetch(wn, buf ^ 1);
        const St &S = st[buf];
        // column pairs j in yv[j % NG]; a position's window 0 needs j = NH .. NG - 1
        float2 yv[NG][4];
        auto get_y = [&](int j, float2 (&v)[4]) {
            const float4 u = *reinterpret_cast<const float4 *>(S.y[j][0][cq]);
            const float4 w = *reinterpret_cast<const float4 *>(S.y[j][1][cq]);
            v[0] = make_float2(u.x, u.y);
            v[1] = make_float2(u.z, u.w);
            v[2] = make_float2(w.x, w.y);
            v[3] = make_float2(w.z, w.w);
        };
#pragma unroll
        for (int j = NH; j < NG - 1; ++j) get_y(j, yv[j]);
        // EDGE 1: the first position of a path's visit, whose cells w < g are
        // columns before it (of another share, or of the previous pair); 2: the
        // last, whose cells w >= g are columns after it.  They count as zero
        // whatever the slots hold
        auto position = [&](int pr, auto edge_tag) {
            constexpr int EDGE = decltype(edge_tag)::value;
            const float *sl = S.g[pr][l];
#pragma unroll
            for (int w = 0; w < NG; ++w) {
                get_y(pr * NG + NG - 1 + w, yv[(NG - 1 + w) % NG]);
                float2 g[NH];
#pragma unroll
                for (int h = 0; h < NH; h += 2) {
                    const float4 v = *reinterpret_cast<const float4 *>(sl + w * NG + 2 * h);
                    g[h] = make_float2(v.x, v.y);
                    g[h + 1] = make_float2(v.z, v.w);
                }
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    if (EDGE == 1 ? w < h : EDGE == 2 && w >= h) g[h].x = 0.f;
                    if (EDGE == 1 ? w < h + NH : EDGE == 2 && w >= h + NH) g[h].y = 0.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        acc[h][c] = fma2(g[h], yv[(NG - 1 + w - h) % NG][c], acc[h][c]);
                }
            }
        };
#pragma unroll 1
        for (int pr = 0; pr < POS; ++pr) {
            const int pos = wk.p + pr;
            if (pos > wk.pe) break;
            if (pos == wk.pb) position(pr, std::integral_constant<int, 1>{});
            else if (pos == wk.pe) position(pr, std::integral_constant<int, 2>{});
            else position(pr, std::integral_constant<int, 0>{});
        }
    }
#pragma unroll
    for (int g = 0; g < NG; ++g) {
        const int real = (l0 + l) * NG + g - a.vrows;
        if (real < 0 || real >= a.nx) continue;
        const int64_t r = opath * a.nx + real;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int n = n0 + 4 * cq + c;
            if (n >= a.N) continue;
            const float v = g < NH ? acc[g % NH][c].x : acc[g % NH][c].y;
            if (a.ksplit > 1) a.partial[((int64_t)ks * a.M + r) * a.N + n] = v;
            else C[r * a.N + n] = v;
        }
    }
}

// The transposed contraction (the column role's increments as output) for lanes
// of 4 or 8 coarse rows, again from the slots as they lie.  A thread owns the NG
// columns of a position and four channels; the cell (row g, column q) is window
// q + g of the position's slot or, past its end, window q + g - NG of the next
// one.  A stage is 32 rows (32 / NG lanes) of one row path, double-buffered by
// cp.async: per lane a thread reads the halves of both slots that it needs (26
// 16-byte loads for NG = 8) and 8 row quads for 256 FMAs, so that the FMAs bound
// it and not the shared memory, where the turned tiles above took three barriers
// and two loads for 16 FMAs.  The upper groups of a window's pairs are kept until
// the lower ones are added: every output takes the rows in band_gemm_kernel's
// order, and the gradients stay bit for bit what they were.
// 8256 pairs (symmetric) of 256-point paths, N = 32: 2.02 -> 1.25 ms a launch.
template <int NG>
struct GcStage {
    static constexpr int LANES = 32 / NG, POS = 128 / NG, THREADS = 8 * POS;
    static constexpr int SLOT = NG * NG, SS = SLOT + 4;   // padded: a warp's 4 positions, 4 bank quads
    float g[LANES][POS + 1][SS];
    float x[32][32];
};

template <int NG>
__global__ void __launch_bounds__(GcStage<NG>::THREADS, 512 / GcStage<NG>::THREADS) band_cols_kernel(GemmArgs a) {
    using St = GcStage<NG>;
    constexpr int NH = NG / 2, POS = St::POS, LANES = St::LANES, SLOT = St::SLOT, NT = St::THREADS;
    constexpr int XV = 1024 / NT;                     // row values a thread stages
    constexpr int SV = SLOT / 4, NV = (POS + 1) * LANES * SV;
    extern __shared__ __align__(16) float gr_sm[];
    St *st = reinterpret_cast<St *>(gr_sm);           // two of them
    const int tid = threadIdx.x, tp = tid >> 3, cq = tid & 7;
    const int64_t b = blockIdx.z / a.ksplit;
    const int ks = blockIdx.z - (int)b * a.ksplit;
    const float *Bm = a.Bm + b * a.b_bstride;
    float *C = a.C + b * a.c_bstride;
    const int TperR = a.TperR1 - 1, tpp = (TperR + POS - 1) / POS;
    // a symmetric Gram's column path j meets j + 1 row paths: the longest first, so
    // that the short ones fill the last wave (1.25 -> 1.11 ms for 128 of them)
    const int64_t blk = blockIdx.x / tpp, opath = a.mode == PM_GRAM_SYM ? a.nB - 1 - blk : blk;
    const int p0 = (int)(blockIdx.x - blk * tpp) * POS;
    const int n0 = blockIdx.y * 32;
    // the share in slices of 32 rows (NG slices a row path)
    const int64_t rhi = a.mode == PM_GRAM_SYM ? opath + 1 : a.nA;
    const int64_t total = rhi * NG;
    const int64_t s_lo = total * ks / a.ksplit, s_hi = total * (ks + 1) / a.ksplit;

    float xr[XV];
    // slice s: its slots into buffer buf (cp.async), its rows' increments into registers
    auto fetch = [&](int64_t s, int buf) {
        const int64_t rp = s / NG;
        const int c0 = (int)(s - rp * NG) * 32;
        const int64_t k = gemm_pair(a, b, rp, opath);
        const float *src = a.band + ((k * a.TperR1 + p0) * 32 + c0 / NG) * (int64_t)SLOT;
        for (int v = tid; v < NV; v += NT) {
            const int sl = v / SV, e = v - sl * SV, pr = sl / LANES, lr = sl % LANES;
            if (p0 + pr <= TperR) cp_async<16>(&st[buf].g[lr][pr][4 * e], src + (pr * 32 + lr) * SLOT + 4 * e);
        }
        cp_commit();
#pragma unroll
        for (int i = 0; i < XV; ++i) {
            const int v = tid + NT * i, real = c0 + (v >> 5) - a.vrows, n = n0 + (v & 31);
            xr[i] = real >= 0 && real < a.nx && n < a.N ? __ldg(Bm + (rp * a.nx + real) * a.N + n) : 0.f;
        }
    };
    float acc[NG][4];
#pragma unroll
    for (int q = 0; q < NG; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[q][c] = 0.f;

    if (s_lo < s_hi) fetch(s_lo, 0);
    int buf = 0;
    for (int64_t s = s_lo; s < s_hi; ++s, buf ^= 1) {
        St &S = st[buf];
#pragma unroll
        for (int i = 0; i < XV; ++i) {
            const int v = tid + NT * i;
            S.x[v >> 5][v & 31] = xr[i];
        }
        cp_wait<0>();
        __syncthreads();   // the stage is complete, and the other buffer's readers are done
        if (s + 1 < s_hi) fetch(s + 1, buf ^ 1);
        const int c0 = (int)(s % NG) * 32;
        if (p0 + tp >= TperR) continue;
        // one lane; MASK: its first `virt` rows are virtual and count as zero whatever the slots hold
        auto lane = [&](int lr, int virt, auto mask_tag) {
            constexpr bool MASK = decltype(mask_tag)::value;
            const float *own = S.g[lr][tp], *nxt = S.g[lr][tp + 1];
            auto row = [&](int g) { return *reinterpret_cast<const float4 *>(&S.x[lr * NG + g][4 * cq]); };
            auto add = [&](int q, float v, int g, const float4 &x) {
                if (MASK && g < virt) v = 0.f;
                acc[q][0] = fmaf(v, x.x, acc[q][0]);
                acc[q][1] = fmaf(v, x.y, acc[q][1]);
                acc[q][2] = fmaf(v, x.z, acc[q][2]);
                acc[q][3] = fmaf(v, x.w, acc[q][3]);
            };
            float hi[NH][NG];   // rows NH + h, until rows 0 .. NH - 1 are added
#pragma unroll
            for (int h = 0; h < NH; h += 2) {
                const float4 xa = row(h), xb = row(h + 1);
#pragma unroll
                for (int w = h; w < NG; ++w) {   // the position's own slot: q = w - g >= 0
                    const float4 v = *reinterpret_cast<const float4 *>(own + w * NG + 2 * h);
                    add(w - h, v.x, h, xa);
                    if (w >= h + 1) add(w - h - 1, v.z, h + 1, xb);
                    if (w >= h + NH) hi[h][w - h - NH] = v.y;
                    if (w >= h + 1 + NH) hi[h + 1][w - h - 1 - NH] = v.w;
                }
#pragma unroll
                for (int w = 0; w < h + 1 + NH; ++w) {   // the next one: q = w - g + NG < NG
                    const float4 v = *reinterpret_cast<const float4 *>(nxt + w * NG + 2 * h);
                    if (w < h) add(w - h + NG, v.x, h, xa);
                    if (w < h + 1) add(w - h - 1 + NG, v.z, h + 1, xb);
                    if (w < h + NH) hi[h][w - h - NH + NG] = v.y;
                    hi[h + 1][w - h - 1 - NH + NG] = v.w;
                }
            }
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const float4 x = row(h + NH);
#pragma unroll
                for (int q = 0; q < NG; ++q) add(q, hi[h][q], h + NH, x);
            }
        };
#pragma unroll 1
        for (int lr = 0; lr < LANES; ++lr) {
            const int virt = a.vrows - (c0 + lr * NG);
            if (virt <= 0) lane(lr, 0, std::false_type{});
            else if (virt < NG) lane(lr, virt, std::true_type{});
        }
    }
    if (p0 + tp >= TperR) return;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
        const int real = (p0 + tp) * NG + q - a.NQV;
        if (real < 0 || real >= a.ny) continue;
        const int64_t r = opath * a.ny + real;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int n = n0 + 4 * cq + c;
            if (n >= a.N) continue;
            if (a.ksplit > 1) a.partial[((int64_t)ks * a.M + r) * a.N + n] = acc[q][c];
            else C[r * a.N + n] = acc[q][c];
        }
    }
}

// ---- the RBF lift's chain rule (Sec. 2.2) ---------------------------------
// With c(p, q) = 1/2 4^-lambda (k(p+1,q+1) - k(p+1,q) - k(p,q+1) + k(p,q)),
// k(i, j) = kappa(x_i, y_j) = exp(-|x_i - y_j|^2 / (2 sigma^2)), the adjoint's
// dk/dc = Gbar gives dL/dk(i, j) = 1/2 4^-lambda W(i, j) with the second
// difference W(i, j) = Gbar(i-1,j-1) - Gbar(i-1,j) - Gbar(i,j-1) + Gbar(i,j)
// (Gbar zero outside the grid), and dk/dx_i = k (y_j - x_i) / sigma^2.  So
// with Wt = 1/2 4^-lambda W k over the points of every pair,
//   dL/dx_i = (sum_j Wt(i,j) y_j - x_i sum_j Wt(i,j)) / sigma^2
// and the mirror for y: a dense contraction of Wt with the points plus the
// row and column sums of Wt.

// C = G B per batch for a dense G read as G[r * ld + k] (or G[k * ld + r] when
// trans), ld a multiple of 4, on the tiles of tile_gemm.cuh; long K ranges split
// across blocks whose partial tiles band_split_sum_kernel adds in order.  G's
// columns are the column paths' points, padded per path from `py` to `py4`
// (zeros): column (path, j) meets B or C row path py + j.  A symmetric Gram's Wt
// holds blocks i <= j only (tri_rb x py4 blocks): the K slices of blocks below
// the diagonal are skipped.  (128 x 128 Gram of 256-point paths, N = 32: 2.9 ms
// on 4 x 4 outputs a thread, 2.4 here.)
struct DenseGemmArgs {
    const float *G;
    int64_t g_ld, g_bstride;
    const float *Bm;
    int64_t b_bstride;
    float *C;
    int64_t c_bstride;
    int64_t M, K;            // padded rows of C (trans) or padded reduction
    int N, trans, ksplit, py, py4;
    int64_t crows;           // unpadded rows of C
    float *partial;
    int64_t tri_rb;
};

template <int NT>
__global__ void __launch_bounds__(TG_THREADS, 2) dense_gemm_kernel(DenseGemmArgs a) {
    using Tile = TileGemm<NT>;
    __shared__ __align__(16) typename Tile::Shared sh;
    const int64_t b = blockIdx.z / a.ksplit;
    const int ks = blockIdx.z - (int)b * a.ksplit;
    const float *G = a.G + b * a.g_bstride;
    const float *Bm = a.Bm + b * a.b_bstride;
    float *C = a.C + b * a.c_bstride;
    const int64_t r0 = (int64_t)blockIdx.x * TG_M;
    const int n0 = blockIdx.y * NT;
    // this block's K range, in whole slices
    int64_t kmin = 0, kmax = a.K;
    if (a.tri_rb > 0) {
        if (!a.trans) kmin = (r0 / a.tri_rb) * a.py4;   // rows of block i: columns of blocks j >= i
        else {                                         // columns of block j: rows of blocks i <= j
            const int64_t rl = (r0 + TG_M - 1 < a.M ? r0 + TG_M - 1 : a.M - 1);
            kmax = (rl / a.py4 + 1) * a.tri_rb;
            if (kmax > a.K) kmax = a.K;
        }
    }
    const int64_t sl0 = kmin / TG_K, nslice = (kmax + TG_K - 1) / TG_K - sl0;
    const int64_t s_lo = sl0 + nslice * ks / a.ksplit, s_hi = sl0 + nslice * (ks + 1) / a.ksplit;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool vec = a.N % 4 == 0 && (reinterpret_cast<uintptr_t>(Bm) & 15) == 0;
    auto load_b = [&](int i, float4 (&v)[NT / 32]) {
#pragma unroll
        for (int u = 0; u < NT / 32; ++u) {
            const int64_t k = (s_lo + i) * TG_K + Tile::template b_line<>(u);
            const int n = n0 + 4 * Tile::template b_quad<>(u);
            v[u] = zero;
            int64_t row = k;
            if (!a.trans) {   // the reduction runs over padded columns
                const int64_t path = k / a.py4;
                const int j = (int)(k - path * a.py4);
                row = j < a.py ? path * a.py + j : -1;
            }
            if (k >= a.K || row < 0) continue;
            const float *p = Bm + row * a.N + n;
            if (vec) {
                if (n < a.N) v[u] = __ldg(reinterpret_cast<const float4 *>(p));
            } else {
                if (n < a.N) v[u].x = p[0];
                if (n + 1 < a.N) v[u].y = p[1];
                if (n + 2 < a.N) v[u].z = p[2];
                if (n + 3 < a.N) v[u].w = p[3];
            }
        }
    };
    Tile t;
    t.clear();
    if (!a.trans) {
        t.template run<true>(sh, (int)(s_hi - s_lo), [&](int i, float4 (&v)[4]) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t r = r0 + Tile::template line<true>(u);
                const int64_t k = (s_lo + i) * TG_K + 4 * Tile::template quad<true>(u);
                v[u] = r < a.M && k < a.K ? __ldcs(reinterpret_cast<const float4 *>(G + r * a.g_ld + k)) : zero;
            }
        }, load_b);
    } else {
        t.template run<false>(sh, (int)(s_hi - s_lo), [&](int i, float4 (&v)[4]) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t k = (s_lo + i) * TG_K + Tile::template line<false>(u);
                const int64_t r = r0 + 4 * Tile::template quad<false>(u);
                v[u] = r < a.M && k < a.K ? __ldcs(reinterpret_cast<const float4 *>(G + k * a.g_ld + r)) : zero;
            }
        }, load_b);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t r = r0 + 8 * (threadIdx.x >> 4) + i;
        if (r >= a.M) continue;
        int64_t row = r;
        if (a.trans) {
            const int64_t path = r / a.py4;
            const int j = (int)(r - path * a.py4);
            if (j >= a.py) continue;
            row = path * a.py + j;
        }
#pragma unroll
        for (int jx = 0; jx < Tile::TN; ++jx) {
            const int n = n0 + Tile::TN * (threadIdx.x & 15) + jx;
            if (n >= a.N) continue;
            if (a.ksplit > 1) a.partial[((int64_t)ks * a.crows + row) * a.N + n] = t.out(i, jx);
            else C[row * a.N + n] = t.out(i, jx);
        }
    }
}

// C = (add ? C : 0) + sum over the splits, in split order (deterministic).
__global__ void band_split_sum_kernel(const float *partial, int ksplit, int64_t MN, int add, float *C) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < MN; v += (int64_t)gridDim.x * blockDim.x) {
        float acc = add ? C[v] : 0.f;
        for (int s = 0; s < ksplit; ++s) acc += partial[s * MN + v];
        C[v] = acc;
    }
}

// Point gradients from increment gradients: x_p enters dx_{p-1} (+) and dx_p
// (-), so dX[path][p] = scale (dinc[p-1] - dinc[p]) (terms outside 0..L-2
// absent).  Overwrites dpts, or adds to it (add).  Both roles in one launch,
// where their outputs share no memory;
// dinc may be the split partials of a contraction, `stride` floats apart, which
// are then added in band_split_sum_kernel's order (one launch less, the same sums).
struct PointsJob {
    const float *dinc;
    int64_t npaths, L, stride;
    int ksplit;
    float *dpts;
};
__global__ void band_points_kernel(PointsJob ja, PointsJob jb, int64_t d, float scale, int add) {
    const int64_t na = ja.npaths * ja.L * d, total = na + jb.npaths * jb.L * d;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < total;
         u += (int64_t)gridDim.x * blockDim.x) {
        const bool isb = u >= na;
        const PointsJob &j = isb ? jb : ja;
        const int64_t v = isb ? u - na : u, c = v % d, row = v / d;
        const int64_t path = row / j.L, p = row - path * j.L;
        const float *di = j.dinc + path * (j.L - 1) * d + c;
        float lo = 0.f, hi = 0.f;
        for (int s = 0; s < j.ksplit; ++s, di += j.stride) {
            if (p >= 1) lo += di[(p - 1) * d];
            if (p < j.L - 1) hi += di[p * d];
        }
        const float g = scale * (lo - hi);
        j.dpts[v] = add ? j.dpts[v] + g : g;
    }
}


// Squared norms of rows of d floats.
__global__ void rbf_norms_kernel(const float *P, int64_t rows, int64_t d, float *out) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int64_t c = 0; c < d; ++c) s = fmaf(P[r * d + c], P[r * d + c], s);
        out[r] = s;
    }
}

// Wt of every pair's (nx+1) x (ny+1) points (see the RBF chain rule above)
// and its row and column sums.  Units are (pair, 128 x 64 point tile).  <x_i,
// y_j> is a tile of tile_gemm.cuh over the channels; |x_i - y_j|^2 = |x_i|^2 +
// |y_j|^2 - 2 <x_i, y_j> (only kappa itself is needed here, so the cancellation
// near x_i = y_j costs an absolute error of about FP32 epsilon times |x|^2).  The
// band slots that hold dk/dc around the tile are staged whole (windows and
// slots padded by one float: the tile's rows and columns then spread over the
// banks), and a thread takes the 9 x 5 values around its 8 x 4 points from
// there.  It is bound by issue slots: per point 16 FMAs' worth at d = 32, about
// 9 for its share of dk/dc, 10 for kappa and the sums.  8 x 4 points a thread
// instead of 4 x 4 and a tile core with vector reads: 128 x 128 Gram of
// 256-point paths, d = 32, 9.6 -> 6.2 ms.
struct RbfWtArgs {
    PairSrc src;             // oriented: rows refine A
    const float *gband;      // dk/dc in the band layout (TperR1 slots per pair)
    float *wt;               // Gram: [row path ia][i] x [column path jb][j], ld = ldw; pairs: [k][i][j]
    float *rsum, *csum;      // sums over j / over i (zeroed before)
    const float *xn, *yn;    // squared norms of the launch's row points and of the column points
    int64_t n_pairs, ldw, a0;
    int TperR1, vrows, NQV, tiles_i, tiles_j, py4;
    float s, scale;          // 1/(2 sigma^2), 1/2 4^-lambda
};
constexpr int RW_TI = TG_M, RW_TJ = 64;

// the staged slots of a tile: lanes (rows), positions (columns), floats a slot
template <int NG>
struct RwStage {
    static constexpr int SL = RW_TI / NG + 1 < 32 ? RW_TI / NG + 1 : 32, SP = RW_TJ / NG + 2;
    static constexpr int WS = NG + 1, SS = NG * WS + 1;
    static constexpr int FLOATS = SL * SP * SS;
};
template <int NG>
constexpr int rw_smem_bytes() {
    constexpr int a = 4 * RwStage<NG>::FLOATS, b = (int)sizeof(typename TileGemm<RW_TJ>::Shared);
    return a + b;
}

template <int NG>
__global__ void __launch_bounds__(TG_THREADS, 2) rbf_wt_kernel(RbfWtArgs a) {
    using Tile = TileGemm<RW_TJ>;
    using St = RwStage<NG>;
    constexpr int SLOT = NG * NG;
    extern __shared__ __align__(16) float rw_sm[];
    typename Tile::Shared &sh = *reinterpret_cast<typename Tile::Shared *>(rw_sm);
    float *stage = rw_sm + sizeof(typename Tile::Shared) / 4;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t d = a.src.d;
    const bool gram = a.src.mode != PM_PAIRS;
    const bool vec = d % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.src.A) | reinterpret_cast<uintptr_t>(a.src.B)) & 15) == 0;
    const int per = a.tiles_i * a.tiles_j, nsl = (int)((d + TG_K - 1) / TG_K);
    for (int64_t u = blockIdx.x; u < a.n_pairs * per; u += gridDim.x) {
        const int64_t k = u / per;
        const int t = (int)(u - k * per);
        const int i0 = (t / a.tiles_j) * RW_TI, j0 = (t % a.tiles_j) * RW_TJ;
        const PairRef pr = pair_ref<true>(a.src, k);
        const int nx = (int)pr.la - 1, ny = (int)pr.lb - 1;   // coarse rows / columns; nx + 1 points
        if (i0 > nx || j0 > ny) continue;   // block-uniform
        const float *xp = (const float *)a.src.A + pr.a_row0 * d;
        const float *yp = (const float *)a.src.B + pr.b_row0 * d;
        __syncthreads();   // the last tile's readers of the stage are done
        // the slots holding dk/dc at (p, q) = (i0 - 1 + pi, j0 - 1 + qj): lanes from
        // l0, positions from s0 (for a position, the lanes are one contiguous run)
        const int Pf = i0 - 1 + a.vrows, Qf = j0 - 1 + a.NQV;
        const int l0 = (Pf < 0 ? 0 : Pf) / NG, s0 = (Qf < 0 ? 0 : Qf) / NG;
        for (int v = tid; v < St::SL * St::SP * (SLOT / 4); v += TG_THREADS) {
            const int sl = v / (SLOT / 4), e = 4 * (v - sl * (SLOT / 4));
            const int sp = sl / St::SL, lr = sl - sp * St::SL;
            if (l0 + lr < 32 && s0 + sp < a.TperR1) {
                const float4 x = __ldcs(reinterpret_cast<const float4 *>(
                    a.gband + ((k * a.TperR1 + s0 + sp) * 32 + l0 + lr) * (int64_t)SLOT + e));
                float *dst = stage + sl * St::SS;
                dst[e / NG * St::WS + e % NG] = x.x;
                dst[(e + 1) / NG * St::WS + (e + 1) % NG] = x.y;
                dst[(e + 2) / NG * St::WS + (e + 2) % NG] = x.z;
                dst[(e + 3) / NG * St::WS + (e + 3) % NG] = x.w;
            }
        }
        // <x_i, y_j>
        auto quad = [&](const float *p, int64_t c) {   // channels c .. c + 3 of the point at p
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (vec) {
                if (c < d) v = __ldg(reinterpret_cast<const float4 *>(p + c));
            } else {
                if (c < d) v.x = __ldg(p + c);
                if (c + 1 < d) v.y = __ldg(p + c + 1);
                if (c + 2 < d) v.z = __ldg(p + c + 2);
                if (c + 3 < d) v.w = __ldg(p + c + 3);
            }
            return v;
        };
        Tile g;
        g.clear();
        g.template run<true, true>(sh, nsl, [&](int sl, float4 (&v)[4]) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = min(i0 + Tile::template line<true>(e), nx);
                v[e] = quad(xp + (int64_t)i * d, (int64_t)sl * TG_K + 4 * Tile::template quad<true>(e));
            }
        }, [&](int sl, float4 (&v)[RW_TJ / 32]) {
#pragma unroll
            for (int e = 0; e < RW_TJ / 32; ++e) {
                const int j = min(j0 + Tile::template b_line<true>(e), ny);
                v[e] = quad(yp + (int64_t)j * d, (int64_t)sl * TG_K + 4 * Tile::template b_quad<true>(e));
            }
        });
        // (the run's barriers also cover the staged slots)
        const int64_t ia = gram ? pr.a_row0 / pr.la - a.a0 : k;
        const int64_t jb = gram ? pr.b_row0 / pr.lb : k;
        const int ib = i0 + 8 * ty, jc = j0 + 4 * tx;   // the thread's first point
        // dk/dc at (p, jc - 1 + e), e < 5, zero outside the grid
        auto row_dc = [&](int p, float (&v)[5]) {
            const int P = p + a.vrows, l = P / NG, gg = P - l * NG;
            const float *base = stage + (l - l0) * St::SS + band_gpos<NG>(gg);
            const bool in = p >= 0 && p < nx;
#pragma unroll
            for (int e = 0; e < 5; ++e) {
                const int q = jc - 1 + e, tq = q + a.NQV + gg;
                v[e] = 0.f;
                if (in && q >= 0 && q < ny) v[e] = base[(tq / NG - s0) * (St::SL * St::SS) + tq % NG * St::WS];
            }
        };
        float yy[4], cs[4] = {0.f, 0.f, 0.f, 0.f}, up[5], dn[5];
#pragma unroll
        for (int j = 0; j < 4; ++j) yy[j] = jc + j <= ny ? a.yn[(gram ? pr.b_row0 : k * (ny + 1)) + jc + j] : 0.f;
        row_dc(ib - 1, up);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int ii = ib + i;
            row_dc(ii, dn);
            float wv[4], rs = 0.f;
            const bool in = ii <= nx;
            const float xx = in ? a.xn[ia * (nx + 1) + ii] : 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float W = up[j] - up[j + 1] - dn[j] + dn[j + 1];
                const float uu = fmaxf(xx + yy[j] - 2.f * g.out(i, j), 0.f);
                wv[j] = in && jc + j <= ny ? a.scale * W * __expf(-a.s * uu) : 0.f;
                rs += wv[j];
                cs[j] += wv[j];
            }
            if (in && jc < a.py4) {   // a path's padding columns get zeros
                float *row = gram ? a.wt + (ia * (nx + 1) + ii) * a.ldw + jb * a.py4
                                  : a.wt + (k * (nx + 1) + ii) * (int64_t)a.py4;
                *reinterpret_cast<float4 *>(row + jc) = make_float4(wv[0], wv[1], wv[2], wv[3]);
            }
            // the row's sum over its 16 threads, one atomic add
#pragma unroll
            for (int o = 1; o < 16; o *= 2) rs += __shfl_xor_sync(FULL, rs, o);
            if (tx == 0 && in) atomicAdd(a.rsum + ia * (nx + 1) + ii, rs);
#pragma unroll
            for (int e = 0; e < 5; ++e) up[e] = dn[e];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            cs[j] += __shfl_xor_sync(FULL, cs[j], 16);
            if ((tid & 16) == 0 && jc + j <= ny) atomicAdd(a.csum + jb * (ny + 1) + jc + j, cs[j]);
        }
    }
}

// out[v] = (add ? out[v] : 0) + f (C1[v] - s1[row] P[v] (+ C2[v] - s2[row] P[v])),
// v = row d + channel: the points' gradients from the contraction and the
// sums (C2, s2: the column role of a symmetric Gram's same paths)
__global__ void rbf_points_kernel(const float *P, int64_t rows, int64_t d, const float *C1, const float *s1,
                                  const float *C2, const float *s2, float f, int add, float *out) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < rows * d;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = v / d;
        float g = C1[v] - s1[row] * P[v];
        if (C2) g += C2[v] - s2[row] * P[v];
        out[v] = add ? out[v] + f * g : f * g;
    }
}

}  // namespace

bool band_geometry(int64_t La, int64_t Lb, int lam, int rows_per_lane, BandPlan &p) {
    if (La < 2 || Lb < 2 || lam < 0 || lam > 3) return false;
    const int64_t S = 1LL << lam;
    const int64_t Ni = S * (La - 1), Nj = S * (Lb - 1);
    int R = 0;
    for (int r : {4, 8, 16})
        if ((rows_per_lane == 0 || rows_per_lane == r) && 32 * r >= Ni && band_has_instance(r, lam)) {
            R = r;
            break;
        }
    if (R == 0) return false;
    const int NG = R >> lam;
    const int64_t Tper = ((Nj + R - 1) / R) * R;
    if (Tper < 2 * R || Tper > (1 << 20)) return false;
    p.R = R;
    p.lam = lam;
    p.NG = NG;
    p.TperR = (int)(Tper / R);
    p.NQ = (int)(Tper / S);
    p.NQV = (int)((Tper - Nj) / S);
    p.vrows = (int)((32 * R - Ni) / S);
    p.slot_floats = (int64_t)32 * NG * NG;
    return true;
}

// workspace: a 256-byte header (the status word of bounded waits), then the band
int64_t band_bytes(const BandPlan &p, int64_t n_pairs) {
    return 256 + (int64_t)sizeof(float) * (n_pairs * p.TperR + 1) * p.slot_floats;
}

// The surface's band-layout values (TperR + 1 slots per pair) after the band:
// their float offset from the band's start, and the whole workspace.
int64_t band_surface_offset(const BandPlan &p, int64_t n_pairs) {
    return ((n_pairs * p.TperR + 1) * p.slot_floats + 63) / 64 * 64;
}
int64_t band_surface_bytes(const BandPlan &p, int64_t n_pairs) {
    return 256 + (int64_t)sizeof(float) *
                     (band_surface_offset(p, n_pairs) + n_pairs * (p.TperR + 1) * p.slot_floats);
}

namespace {
// The band coefficients: the FP32 kernel of band_coef.cu, or on request
// (coef_path 3, d <= 64, linear kernel) the tcgen05 kernel, whose one block per
// SM serialises staging, MMAs and the scattered band write-back (measured on
// the 128 x 128 MMD Gram, d = 32: 4.8 ms against 2.3).
cudaError_t launch_band_coef(const BandCoefArgs &c, const BandPlan &p, int sms, int *status, cudaStream_t st,
                             int coef_path) {
    if (c.src.kernel == SIGK_KERNEL_LINEAR && coef_path == 3 && c.src.d <= 64) {
        if (p.NG == 8) return launch_coef_tc5<8>(c, sms, status, st);
        if (p.NG == 4) return launch_coef_tc5<4>(c, sms, status, st);
        return launch_coef_tc5<2>(c, sms, status, st);
    }
    return launch_band_coefs(c.src, p, c.n_pairs, c.band, sms, st);
}
}  // namespace

cudaError_t launch_band_f32(const PairSrc &src, const BandPlan &p, int64_t n_pairs, float *out,
                            void *ws, cudaStream_t st, int coef_path, float *surf, int64_t s_pair,
                            int64_t s_a, int64_t s_b) {
    if (n_pairs <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    int *status = (int *)ws;
    float *band = (float *)((unsigned char *)ws + 256);
    if ((e = cudaMemsetAsync(status, 0, sizeof(int), st)) != cudaSuccess) return e;
    BandCoefArgs c;
    c.src = src;
    c.n_pairs = n_pairs;
    c.TperR = p.TperR;
    c.NQ = p.NQ;
    c.NQV = p.NQV;
    c.vrows = p.vrows;
    c.scale = 0.5f / (float)(1 << (2 * p.lam));
    c.band = band;
    if ((e = launch_band_coef(c, p, sms, status, st, coef_path)) != cudaSuccess) return e;

    const int per_sm = band_occupancy_of(p.R, p.lam);
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t warps = (int64_t)sms * per_sm * BAND_WARPS;
    BandArgs a;
    memset(&a, 0, sizeof(a));
    a.src = src;
    a.out = out;
    a.band = band;
    a.n_pairs = n_pairs;
    a.ppw = (n_pairs + warps - 1) / warps;
    a.TperR = p.TperR;
    // the surface's band-layout values follow the coefficient band in the workspace
    a.sband = surf ? band + band_surface_offset(p, n_pairs) : nullptr;
    const int64_t nwarps = (n_pairs + a.ppw - 1) / a.ppw;
    const int grid = (int)((nwarps + BAND_WARPS - 1) / BAND_WARPS);
    bool launched = false;
#define X(r, l, mb)                                                                  \
    if (p.R == r && p.lam == l) {                                                    \
        if (surf)                                                                    \
            chain_band_kernel<r, l, mb, false, true><<<grid, BAND_WARPS * 32, 0, st>>>(a); \
        else                                                                         \
            chain_band_kernel<r, l, mb, false><<<grid, BAND_WARPS * 32, 0, st>>>(a);       \
        launched = true;                                                             \
    }
    SIGK_BAND_CASES(X)
#undef X
    if (!launched) return cudaErrorInvalidValue;
    if ((e = cudaGetLastError()) != cudaSuccess || !surf) return e;
    return launch_surface_unpack(src, p, n_pairs, a.sband, surf, s_pair, s_a, s_b, st);
}

cudaError_t launch_surface_unpack(const PairSrc &src, const BandPlan &p, int64_t n_pairs, const float *sband,
                                  float *surf, int64_t s_pair, int64_t s_a, int64_t s_b, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    // the surface from the band layout into [pair][L][M]
    BandGbarArgs gb;
    memset(&gb, 0, sizeof(gb));
    gb.src = src;
    gb.gband = sband;
    gb.gbar = surf;
    gb.n_pairs = n_pairs;
    gb.TperR = p.TperR;
    gb.NQV = p.NQV;
    gb.vrows = p.vrows;
    gb.nx = (int)(src.La - 1);
    gb.ny = (int)(src.Lb - 1);
    gb.s_pair = s_pair;
    gb.s_a = s_a;
    gb.s_b = s_b;
    gb.q_off = p.lam == 0 ? 1 : 0;
    const int64_t tasks = n_pairs * gb_groups(p.TperR, true, p.NG);
    const int ggrid = (int)(tasks < (int64_t)sms * 8 ? tasks : (int64_t)sms * 8);
    if (p.NG == 8) band_gbar_kernel<8><<<ggrid, GB_THREADS, 0, st>>>(gb);
    else if (p.NG == 4) band_gbar_kernel<4><<<ggrid, GB_THREADS, 0, st>>>(gb);
    else band_gbar_kernel<2><<<ggrid, GB_THREADS, 0, st>>>(gb);
    return cudaGetLastError();
}

}  // namespace sigk

// ---- the band backward -------------------------------------------------------

namespace sigk {

namespace {

template <int R, int LAM>
cudaError_t launch_adj(const BandAdjArgs &a, int64_t nwarps, cudaStream_t st) {
    const int smem = (int)sizeof(float) * BAND_WARPS * adj_warp_floats<R, LAM>();
    auto kern = chain_band_adj_kernel<R, LAM>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int64_t grid = (nwarps + BAND_WARPS - 1) / BAND_WARPS;
    kern<<<(int)grid, BAND_WARPS * 32, smem, st>>>(a);
    return cudaGetLastError();
}

int64_t up4(int64_t v) { return (v + 3) / 4 * 4; }

// Float counts of the backward's workspace regions for a launch of nbp pairs
// (Gram: whole rows of nb pairs).  Checkpoint and last-row regions are sized
// for any pairs-per-warp split (they are checked against the actual split at
// launch).
struct BwdRegions {
    int64_t band, gbar, ckpt, exitk, botq, incA, incB, dincA, dincB, part, gband, rsum;
    int64_t total() const {
        return band + gbar + ckpt + exitk + botq + incA + incB + dincA + dincB + part + gband + rsum;
    }
};

// dense: whether a Gram's dk/dc is unpacked into a dense matrix for the
// tensor-core contraction (coef_path 3); the FP32 contraction reads the band
bool bwd_dense_gbar(const PairSrc &src, int coef_path) {
    const bool gram = src.mode == PM_GRAM || src.mode == PM_GRAM_SYM;
    return gram && src.kernel == SIGK_KERNEL_LINEAR && coef_path == 3 && chain_gemm_tc5_ok(1, 1, (int)src.d);
}

BwdRegions bwd_regions(const PairSrc &src, const BandPlan &p, int64_t nbp, int coef_path) {
    const int64_t nx = src.La - 1, ny = src.Lb - 1, d = src.d;
    const bool sym = src.mode == PM_GRAM_SYM;
    const bool gram = src.mode == PM_GRAM || sym;
    const int64_t nA = sym ? src.nb : gram ? (nbp + src.nb - 1) / src.nb : nbp;
    const int64_t nB = gram ? src.nb : nbp;
    BwdRegions r;
    r.band = up4(band_bytes(p, nbp) / (int64_t)sizeof(float));
    r.gbar = bwd_dense_gbar(src, coef_path) ? up4(nA * nx * nB * ny) : 0;
    r.ckpt = ((nbp + 1) * ((2 * (int64_t)p.TperR + 32 + BAND_CK) / BAND_CK) + 1) * 32 * 2 * p.R;
    r.exitk = (nbp + 1) * 32 * (int64_t)p.R;
    r.botq = up4((nbp + 1) * ((2 * (int64_t)p.TperR + 32) * p.R + 4));
    r.incA = up4(nA * nx * d);
    r.incB = up4(nB * ny * d);
    r.dincA = r.incA;
    r.dincB = r.incB;
    // split-K partial tiles of the Gram's contractions
    r.part = gram ? up4((int64_t)GEMM_MAX_SPLIT * (nA * nx > nB * ny ? nA * nx : nB * ny) * d) : 0;
    r.rsum = 0;
    if (src.kernel == SIGK_KERNEL_RBF) {
        // the lift works on points: Wt of every pair (dense, in gbar), the
        // contractions' results (dinc), the row and column sums; no increments
        const int64_t px = nx + 1, py = ny + 1;
        r.gbar = nA * px * nB * up4(py);
        if (!gram) r.gbar = nbp * px * up4(py);
        r.incA = r.incB = 0;
        r.dincA = up4(nA * px * d);
        r.dincB = up4(nB * py * d);
        r.part = gram ? up4((int64_t)GEMM_MAX_SPLIT * (nA * px > nB * py ? nA * px : nB * py) * d) : 0;
        r.rsum = 2 * (up4(nA * px) + up4(nB * py));   // and the points' squared norms
    }
    // the adjoint's dk/dc in the band layout: TperR + 1 slots per pair
    r.gband = up4(nbp * ((int64_t)p.TperR + 1) * 32 * p.NG * p.NG);
    return r;
}

}  // namespace

int64_t band_bwd_batch(const PairSrc &src, const BandPlan &p, int64_t n, int64_t cap_bytes,
                       int64_t &bytes, int coef_path) {
    if (src.mode == PM_GRAM_SYM) {   // one launch: every pair involves the same paths
        bytes = bwd_regions(src, p, n, coef_path).total() * (int64_t)sizeof(float);
        return n;
    }
    // whole Gram rows per launch: each launch owns its row paths' gradients
    const int64_t unit = src.mode == PM_GRAM ? src.nb : 1;
    int64_t units = (n + unit - 1) / unit;
    int64_t nb = n;
    bytes = bwd_regions(src, p, nb, coef_path).total() * (int64_t)sizeof(float);
    while (units > 1 && bytes > cap_bytes) {
        units = (units + 1) / 2;
        nb = units * unit < n ? units * unit : n;
        bytes = bwd_regions(src, p, nb, coef_path).total() * (int64_t)sizeof(float);
    }
    return nb;
}

// The RBF lift's chain rule for one launch of the band backward (pairs
// kbase .. kbase + m of the oriented src; Gram: row paths a0 .. a0 + nA
// against all nB column paths): Wt and its sums, the dense contractions
// CX = Wt Y and CY = Wt^T X, then the points' gradients.  dA is overwritten
// (or added to: add); dB likewise on the first launch and added to after.
cudaError_t rbf_chain_rule(const PairSrc &src, const BandPlan &p, int64_t m, int64_t a0, int64_t nA, int64_t nB,
                           int64_t kb, const float *gband, float *wt, float *CX, float *CY, float *rsum,
                           float *part, float *dA, float *dB, bool add, int sms, cudaStream_t st) {
    const bool sym = src.mode == PM_GRAM_SYM;
    const bool gram = src.mode == PM_GRAM || sym;
    const int64_t d = src.d, px = src.La, py = src.Lb;   // points per path
    const int64_t nrow = gram ? nA : m, ncol = gram ? nB : m;
    float *csum = rsum + up4(nrow * px);
    cudaError_t e;
    if ((e = cudaMemsetAsync(rsum, 0, sizeof(float) * (size_t)(up4(nrow * px) + ncol * py), st)) != cudaSuccess)
        return e;
    // a symmetric Gram stores pairs i <= j: the blocks below the diagonal stay zero
    const int64_t py4 = up4(py);
    if (sym && (e = cudaMemsetAsync(wt, 0, sizeof(float) * (size_t)(nA * px * nB * py4), st)) != cudaSuccess)
        return e;
    const float *Apts = (const float *)src.A + (gram ? a0 : src.kbase) * px * d;
    const float *Bpts = sym ? (const float *)src.A : (const float *)src.B + (gram ? 0 : src.kbase) * py * d;
    float *xn = csum + up4(ncol * py), *yn = xn + up4(nrow * px);
    rbf_norms_kernel<<<(unsigned)((nrow * px + 255) / 256 < sms * 8 ? (nrow * px + 255) / 256 : sms * 8), 256, 0, st>>>(
        Apts, nrow * px, d, xn);
    rbf_norms_kernel<<<(unsigned)((ncol * py + 255) / 256 < sms * 8 ? (ncol * py + 255) / 256 : sms * 8), 256, 0, st>>>(
        Bpts, ncol * py, d, yn);
    RbfWtArgs w;
    w.src = src;
    w.gband = gband;
    w.wt = wt;
    w.rsum = rsum;
    w.csum = csum;
    w.n_pairs = m;
    w.xn = xn;
    w.yn = yn;
    w.py4 = (int)py4;
    w.ldw = gram ? nB * py4 : py4;
    w.a0 = a0;
    w.TperR1 = p.TperR + 1;
    w.vrows = p.vrows;
    w.NQV = p.NQV;
    w.tiles_i = (int)((px + RW_TI - 1) / RW_TI);
    w.tiles_j = (int)((py + RW_TJ - 1) / RW_TJ);
    w.s = (float)(0.5 / (src.sigma * src.sigma));
    w.scale = 0.5f / (float)(1 << (2 * p.lam));
    int64_t grid = m * w.tiles_i * w.tiles_j;
    if (grid > (int64_t)sms * 2) grid = (int64_t)sms * 2;
    auto go = [&](auto kern, int smem) {
        cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (r != cudaSuccess) return r;
        kern<<<(int)grid, TG_THREADS, smem, st>>>(w);
        return cudaGetLastError();
    };
    if (p.NG == 8) e = go(rbf_wt_kernel<8>, rw_smem_bytes<8>());
    else if (p.NG == 4) e = go(rbf_wt_kernel<4>, rw_smem_bytes<4>());
    else e = go(rbf_wt_kernel<2>, rw_smem_bytes<2>());
    if (e != cudaSuccess) return e;
    // the contractions
    DenseGemmArgs g1;
    memset(&g1, 0, sizeof(g1));
    g1.G = wt;
    g1.N = (int)d;
    DenseGemmArgs g2 = g1;
    g1.Bm = Bpts;
    g1.C = CX;
    g1.trans = 0;
    g2.Bm = Apts;
    g2.C = CY;
    g2.trans = 1;
    g1.py = g2.py = (int)py;
    g1.py4 = g2.py4 = (int)py4;
    int64_t batches = 1;
    if (gram) {
        g1.g_ld = g2.g_ld = nB * py4;
        g1.M = nA * px; g1.K = nB * py4;
        g2.M = nB * py4; g2.K = nA * px;
        g1.crows = nA * px; g2.crows = nB * py;
        g1.tri_rb = g2.tri_rb = sym ? px : 0;
    } else {
        batches = m;
        g1.g_ld = g2.g_ld = py4;
        g1.g_bstride = g2.g_bstride = px * py4;
        g1.b_bstride = py * d; g2.b_bstride = px * d;
        g1.c_bstride = px * d; g2.c_bstride = py * d;
        g1.M = px; g1.K = py4;
        g2.M = py4; g2.K = px;
        g1.crows = px; g2.crows = py;
    }
    const int nt = d > 32 ? 64 : 32;
    auto split = [&](const DenseGemmArgs &g) {
        if (!gram) return 1;
        const int64_t tiles = ((g.M + TG_M - 1) / TG_M) * ((d + nt - 1) / nt);
        int64_t ksp = (4 * (int64_t)sms + tiles - 1) / tiles;
        const int64_t nsl = (g.K + TG_K - 1) / TG_K;
        if (ksp > nsl / 4) ksp = nsl / 4;
        if (ksp > GEMM_MAX_SPLIT) ksp = GEMM_MAX_SPLIT;
        return (int)(ksp < 1 ? 1 : ksp);
    };
    g1.ksplit = split(g1);
    g2.ksplit = split(g2);
    g1.partial = g2.partial = part;
    const bool want_b = dB || sym;
    for (int pass = 0; pass < (want_b ? 2 : 1); ++pass) {
        const DenseGemmArgs &g = pass == 0 ? g1 : g2;
        const dim3 gd((unsigned)((g.M + TG_M - 1) / TG_M), (unsigned)((d + nt - 1) / nt),
                      (unsigned)(batches * g.ksplit));
        if (nt == 64) dense_gemm_kernel<64><<<gd, TG_THREADS, 0, st>>>(g);
        else dense_gemm_kernel<32><<<gd, TG_THREADS, 0, st>>>(g);
        if (g.ksplit > 1) band_split_sum_kernel<<<sms * 4, 256, 0, st>>>(part, g.ksplit, g.crows * d, 0, g.C);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // the points
    const float f = (float)(1.0 / (src.sigma * src.sigma));
    if (dA) {
        float *out = dA + (gram ? a0 : src.kbase) * px * d;
        rbf_points_kernel<<<sms * 4, 256, 0, st>>>(Apts, nrow * px, d, CX, rsum, sym ? CY : nullptr,
                                                   sym ? csum : nullptr, f, add ? 1 : 0, out);
    }
    if (dB && !sym) {
        float *out = dB + (gram ? 0 : src.kbase) * py * d;
        rbf_points_kernel<<<sms * 4, 256, 0, st>>>(Bpts, ncol * py, d, CY, csum, nullptr, nullptr, f,
                                                   (add || (gram && kb > 0)) ? 1 : 0, out);
    }
    return cudaGetLastError();
}

cudaError_t launch_band_bwd_f32(const PairSrc &src0, const BandPlan &p, int64_t n, int64_t nbp,
                                const float *gout, float *dA, float *dB, void *ws, cudaStream_t st,
                                int coef_path, float *out, bool add) {
    if (n <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int per_sm = band_occupancy_of(p.R, p.lam);
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    // symmetric Gram: pairs (i, j), i <= j, of one batch; dA gets the
    // derivative through both arguments (dB must be null)
    const bool sym = src0.mode == PM_GRAM_SYM;
    const bool gram = src0.mode == PM_GRAM || sym;
    if (sym && (dB || nbp != n)) return cudaErrorInvalidValue;
    const int64_t nx = src0.La - 1, ny = src0.Lb - 1, d = src0.d;
    const float scale = 0.5f / (float)(1 << (2 * p.lam));
    const BwdRegions rg = bwd_regions(src0, p, nbp, coef_path);
    float *w = (float *)ws;
    int *status = (int *)ws;
    float *band = w + 64;   // after the 256-byte status header
    float *gbar = w + rg.band;
    float *ckpt = gbar + rg.gbar;
    float *exitk = ckpt + rg.ckpt;
    float *botq = exitk + rg.exitk;
    float *incA = botq + rg.botq;
    float *incB = incA + rg.incA;
    float *dincA = incB + rg.incB;
    float *dincB = dincA + rg.dincA;
    float *part = dincB + rg.dincB;
    float *gband = part + rg.part;
    float *rsum = gband + rg.gband;   // the RBF lift's row sums, then its column sums
    const bool rbf = src0.kernel == SIGK_KERNEL_RBF;
    const int64_t nBall = gram ? src0.nb : 0;
    if (rbf && (e = cudaMemsetAsync(status, 0, sizeof(int), st)) != cudaSuccess) return e;
    for (int64_t kb = 0; kb < n; kb += nbp) {
        const int64_t m = n - kb < nbp ? n - kb : nbp;
        PairSrc src = src0;
        src.kbase = src0.kbase + kb;
        const int64_t a0 = sym ? 0 : gram ? src.kbase / src0.nb : src.kbase;   // first row path
        const int64_t nA = sym ? src0.nb : gram ? m / src0.nb : m;
        // 1. increments of this launch's paths (a Gram's column paths, which every
        // launch uses, with the first one's; a symmetric one has no others), and coefficients
        if (!rbf) {
            const bool b = !sym && (!gram || kb == 0);
            const IncJob ja = {(const float *)src.A + a0 * src.La * d, nA, src.La, incA};
            const IncJob jb = {(const float *)src.B + (gram ? 0 : src.kbase * src.Lb * d), !b ? 0 : gram ? nBall : m,
                               src.Lb, incB};
            band_inc_kernel<<<sms * 4, 256, 0, st>>>(ja, jb, d, kb == 0 ? status : nullptr);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        BandCoefArgs c;
        c.src = src;
        c.n_pairs = m;
        c.TperR = p.TperR;
        c.NQ = p.NQ;
        c.NQV = p.NQV;
        c.vrows = p.vrows;
        c.scale = scale;
        c.band = band;
        if ((e = launch_band_coef(c, p, sms, status, st, coef_path)) != cudaSuccess) return e;
        // 2. the forward sweep, keeping what the adjoint needs
        const int64_t warps = (int64_t)sms * per_sm * BAND_WARPS;
        BandArgs f;
        memset(&f, 0, sizeof(f));
        f.src = src;
        f.band = band;
        f.n_pairs = m;
        f.ppw = (m + warps - 1) / warps;
        f.TperR = p.TperR;
        const int64_t nwarps = (m + f.ppw - 1) / f.ppw;
        const int64_t tm = f.ppw * p.TperR + 32;
        f.nck = (int)((tm + BAND_CK - 1) / BAND_CK);
        f.bq_stride = up4(tm * p.R + 1);
        if (nwarps * f.nck * 32 * 2 * p.R > rg.ckpt || nwarps * f.bq_stride > rg.botq)
            return cudaErrorInvalidValue;   // the workspace bound does not hold (cannot happen)
        f.ckpt = ckpt;
        f.exitk = exitk;
        f.botq = botq;
        f.out = out;   // the values too, when the caller asks (sigk_gram_value_and_grad)
        const int fgrid = (int)((nwarps + BAND_WARPS - 1) / BAND_WARPS);
        bool launched = false;
#define X(r, l, mb)                                                              \
        if (p.R == r && p.lam == l) {                                            \
            chain_band_kernel<r, l, mb, true><<<fgrid, BAND_WARPS * 32, 0, st>>>(f); \
            launched = true;                                                     \
        }
        SIGK_BAND_CASES(X)
#undef X
        if (!launched) return cudaErrorInvalidValue;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // 3. the adjoint sweep: dk/dc into gbar
        BandAdjArgs ad;
        ad.src = src;
        ad.band = band;
        ad.ckpt = ckpt;
        ad.exitk = exitk;
        ad.botq = botq;
        ad.nck = f.nck;
        ad.bq_stride = f.bq_stride;
        ad.gout = gout;
        ad.gband = gband;
        ad.n_pairs = m;
        ad.ppw = f.ppw;
        ad.TperR = p.TperR;
        ad.NQ = p.NQ;
        ad.NQV = p.NQV;
        ad.vrows = p.vrows;
        ad.nx = (int)nx;
        ad.ny = (int)ny;
        launched = false;
#define X(r, l, mb)                                                  \
        if (p.R == r && p.lam == l) {                                \
            if ((e = launch_adj<r, l>(ad, nwarps, st)) != cudaSuccess) return e; \
            launched = true;                                         \
        }
        SIGK_BAND_CASES(X)
#undef X
        if (!launched) return cudaErrorInvalidValue;
        if (rbf) {
            // the RBF lift: the chain rule through kappa over the points
            if ((e = rbf_chain_rule(src, p, m, a0, nA, nBall, kb, gband, gbar, dincA, dincB, rsum, part, dA, dB,
                                    add, sms, st)) != cudaSuccess)
                return e;
            continue;
        }
        // a Gram's contractions on the tensor cores (split-TF32) with the
        // tcgen05 path (coef_path 3), else on the FP32 pipe.  The tensor-core
        // contraction matches the FP32 one's accuracy but measured slower on
        // the 128 x 128 MMD Gram (2.6 against 1.5 ms a launch): its chunks run
        // in lockstep (copy, split, MMAs, read-back behind block barriers)
        const bool tc = bwd_dense_gbar(src0, coef_path);
        // 3b. dk/dc from the band layout into the dense Gbar (the tensor-core
        // contraction reads it; the FP32 one reads the band layout itself)
        if (tc) {
            // blocks below the diagonal of a symmetric Gram's dense dk/dc stay zero
            if (sym && cudaMemsetAsync(gbar, 0, sizeof(float) * rg.gbar, st) != cudaSuccess) return cudaErrorUnknown;
            BandGbarArgs gb;
            memset(&gb, 0, sizeof(gb));   // s_pair = 0: the dense Gbar, not the surface
            gb.src = src;
            gb.gband = gband;
            gb.gbar = gbar;
            gb.g_ld = gram ? nBall * ny : ny;
            gb.a_first = a0;
            gb.gram = gram ? 1 : 0;
            gb.n_pairs = m;
            gb.TperR = p.TperR;
            gb.NQV = p.NQV;
            gb.vrows = p.vrows;
            gb.nx = (int)nx;
            gb.ny = (int)ny;
            const int64_t tasks = m * gb_groups(p.TperR, false, p.NG);
            const int ggrid = (int)(tasks < (int64_t)sms * 8 ? tasks : (int64_t)sms * 8);
            if (p.NG == 8) band_gbar_kernel<8><<<ggrid, GB_THREADS, 0, st>>>(gb);
            else if (p.NG == 4) band_gbar_kernel<4><<<ggrid, GB_THREADS, 0, st>>>(gb);
            else band_gbar_kernel<2><<<ggrid, GB_THREADS, 0, st>>>(gb);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        // 4. chain rule: dinc_A = gbar inc_B, dinc_B (+)= gbar^T inc_A
        GemmArgs g1;
        memset(&g1, 0, sizeof(g1));
        g1.G = gbar;
        g1.Bm = sym ? incA : incB;
        g1.C = dincA;
        g1.N = (int)d;
        g1.trans = 0;
        g1.tri_rb = sym ? nx : 0;
        g1.tri_cb = sym ? ny : 0;
        GemmArgs g2 = g1;
        g2.Bm = incA;
        g2.C = dincB;
        g2.trans = 1;
        int64_t batches;
        if (gram) {
            batches = 1;
            g1.g_ld = g2.g_ld = nBall * ny;
            g1.M = nA * nx; g1.K = nBall * ny;
            g2.M = nBall * ny; g2.K = nA * nx;
            g1.nA = g2.nA = nA;
            g1.nB = g2.nB = nBall;
        } else {
            batches = m;
            g1.b_bstride = ny * d; g2.b_bstride = nx * d;
            g1.c_bstride = nx * d; g2.c_bstride = ny * d;
            g1.M = nx; g1.K = ny;
            g2.M = ny; g2.K = nx;
            g1.nA = g2.nA = 1;
            g1.nB = g2.nB = 1;
        }
        // output tiles: 128 band coordinates of one output path (band rows,
        // or band columns when trans) by 32 channels
        const int64_t BHr = 32 * (int64_t)p.NG, NQc = (int64_t)p.TperR * p.NG;
        const int64_t tiles1 = (gram ? g1.nA : 1) * ((BHr + GT_M - 1) / GT_M);
        const int64_t tiles2 = (gram ? g2.nB : 1) * ((NQc + GT_M - 1) / GT_M);
        // a Gram's contractions have long reductions: split them to about four
        // blocks per SM, the partial tiles summed in a fixed order.  The Gram's
        // column-path gradients add up over launches.
        auto split = [&](int64_t tiles, int64_t nsl) {
            if (!gram) return 1;
            tiles *= (d + GT_N - 1) / GT_N;
            int64_t ksp = (4 * (int64_t)sms + tiles - 1) / tiles;
            if (ksp > nsl / 4) ksp = nsl / 4;
            if (ksp > GEMM_MAX_SPLIT) ksp = GEMM_MAX_SPLIT;
            return (int)(ksp < 1 ? 1 : ksp);
        };
        g1.ksplit = split(tiles1, nBall * ((NQc + GT_K - 1) / GT_K));
        g2.ksplit = split(tiles2, nA * (BHr / GT_K));
        g1.partial = g2.partial = part;
        const bool add_b = (gram && kb > 0) || sym;
        if (sym) g2.C = dincA;   // column-role gradients of the same paths: add them to the row role's
        // the split sum writes the result; an unsplit contraction that must add goes through it too
        if (add_b && g2.ksplit == 1) g2.ksplit = 2;
        const dim3 gd1((unsigned)tiles1, (unsigned)((d + GT_N - 1) / GT_N), (unsigned)(batches * g1.ksplit));
        const dim3 gd2((unsigned)tiles2, (unsigned)((d + GT_N - 1) / GT_N), (unsigned)(batches * g2.ksplit));
        // the FP32 contractions gather dk/dc from the band layout
        g1.band = g2.band = gband;
        g1.mode = g2.mode = src.mode;
        g1.nb = g2.nb = src0.nb;
        g1.a0 = g2.a0 = a0;
        g1.kbase = g2.kbase = src.kbase;
        g1.TperR1 = g2.TperR1 = p.TperR + 1;
        g1.vrows = g2.vrows = p.vrows;
        g1.NQV = g2.NQV = p.NQV;
        g1.nx = g2.nx = (int)nx;
        g1.ny = g2.ny = (int)ny;
        // as the slots lie for 4 and 8 rows a lane, through turned tiles for 2
        auto go = [&](auto kern, int threads, size_t smem, const dim3 &gd, const GemmArgs &ga) {
            if (smem > 0) {
                cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (r != cudaSuccess) return r;
            }
            kern<<<gd, threads, smem, st>>>(ga);
            return cudaGetLastError();
        };
        auto as_chain = [&](const GemmArgs &ga, int add) {
            ChainGemm cg;
            cg.G = ga.G;
            cg.g_ld = ga.g_ld;
            cg.trans = ga.trans;
            cg.Bm = ga.Bm;
            cg.C = ga.C;
            cg.M = ga.M;
            cg.K = ga.K;
            cg.N = ga.N;
            cg.add = add;
            cg.tri_rb = ga.tri_rb;
            cg.tri_cb = ga.tri_cb;
            return cg;
        };
        if (dA) {
            if (tc) {
                if ((e = launch_chain_gemm_tc5(as_chain(g1, 0), status, st)) != cudaSuccess) return e;
            } else {
                if (p.NG == 8) e = go(band_rows_kernel<8>, GrStage<8>::THREADS, 2 * sizeof(GrStage<8>), gd1, g1);
                else if (p.NG == 4) e = go(band_rows_kernel<4>, GrStage<4>::THREADS, 2 * sizeof(GrStage<4>), gd1, g1);
                else e = go(band_gemm_kernel<2>, 256, 0, gd1, g1);
                if (e != cudaSuccess) return e;
                if (g1.ksplit > 1)
                    band_split_sum_kernel<<<sms * 4, 256, 0, st>>>(part, g1.ksplit, g1.M * d, 0, dincA);
            }
        }
        if (dB || sym) {
            if (tc) {
                if ((e = launch_chain_gemm_tc5(as_chain(g2, add_b ? 1 : 0), status, st)) != cudaSuccess) return e;
            } else {
                if (p.NG == 8) e = go(band_cols_kernel<8>, GcStage<8>::THREADS, 2 * sizeof(GcStage<8>), gd2, g2);
                else if (p.NG == 4) e = go(band_cols_kernel<4>, GcStage<4>::THREADS, 2 * sizeof(GcStage<4>), gd2, g2);
                else e = go(band_gemm_kernel<2>, 256, 0, gd2, g2);
                if (e != cudaSuccess) return e;
                if (g2.ksplit > 1 && add_b)
                    band_split_sum_kernel<<<sms * 4, 256, 0, st>>>(part, g2.ksplit, g2.M * d, 1, g2.C);
                else if (g2.ksplit > 1 && kb + m < n)   // the last launch's are summed by the point gradients
                    band_split_sum_kernel<<<sms * 4, 256, 0, st>>>(part, g2.ksplit, g2.M * d, 0, g2.C);
            }
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // 5. point gradients (a Gram's column paths' with the last launch's)
        PointsJob ja = {dincA, dA ? nA : 0, src.La, 0, 1, dA ? dA + a0 * src.La * d : nullptr};
        PointsJob jb = {dincB, 0, src.Lb, 0, 1, dB};
        if (dB && !gram) {
            jb.npaths = m;
            jb.dpts = dB + src.kbase * src.Lb * d;
        } else if (dB && kb + m >= n) {
            jb.npaths = nBall;
            if (!tc && !add_b && g2.ksplit > 1) {
                jb.dinc = part;
                jb.ksplit = g2.ksplit;
                jb.stride = g2.M * d;
            }
        }
        // outputs that share memory (one buffer that collects both derivatives of a
        // Gram of X with itself) take the roles one after the other
        const float *da = ja.dpts, *db = jb.dpts;
        const bool shared = ja.npaths && jb.npaths && da < db + jb.npaths * jb.L * d && db < da + ja.npaths * ja.L * d;
        if (shared) {
            PointsJob none = jb;
            none.npaths = 0;
            band_points_kernel<<<sms * 4, 256, 0, st>>>(ja, none, d, scale, add);
            ja.npaths = 0;
        }
        if (ja.npaths || jb.npaths) band_points_kernel<<<sms * 4, 256, 0, st>>>(ja, jb, d, scale, add);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}


}  // namespace sigk
