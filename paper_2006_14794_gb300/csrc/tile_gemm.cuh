// The FP32 tile of the chain rules' contractions: C[128][NT] = sum over k of
// G(m, k) B(k, n), by blocks of 256 threads, 8 x NT/16 outputs a thread.
//
// What bounds it: the FP32 pipe, 4 NT/16 packed FMAs (rows m, m + 1 of a pair in
// one float2) for two float4s of G, both broadcast, and one vector of B a k,
// about 4 shared-memory wavefronts against 8 cycles of FMAs at NT = 64.  Slices
// of 32 k are double-buffered: the next one is loaded into registers while the
// current one is used, one barrier a slice.  G may lie with k contiguous (its
// float4s are turned in shared memory) or with m contiguous; either way element
// (k, m) is kept at [k][m ^ 4 ((k / 4) % 8)], so the turned stores of a warp hit
// 32 banks and the float4 reads stay whole.  B likewise (element (k, n) at [k][n
// ^ 4 ((k / 4) % 8)]).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace sigk {

constexpr int TG_M = 128, TG_K = 32, TG_THREADS = 256;

template <int NT>
struct TileGemm {
    static constexpr int TN = NT / 16;   // columns a thread
    float2 acc[4][TN];                   // rows 8 ty + 2 i, + 1

    struct Shared {
        float g[2][TG_K][TG_M];
        float b[2][TG_K][NT];
    };

    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int n = 0; n < TN; ++n) acc[i][n] = make_float2(0.f, 0.f);
    }
    // the thread's share of a slice's G: float4 i is row (k contiguous) or
    // slice line (m contiguous) line(i), float4 quad(i) of it
    template <bool KCONT>
    static __device__ __forceinline__ int line(int i) {
        const int v = threadIdx.x + TG_THREADS * i;
        return KCONT ? v >> 3 : v >> 5;
    }
    template <bool KCONT>
    static __device__ __forceinline__ int quad(int i) {
        const int v = threadIdx.x + TG_THREADS * i;
        return KCONT ? v & 7 : v & 31;
    }
    template <bool KCONT>
    static __device__ __forceinline__ void put_g(Shared &s, int buf, const float4 (&v)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int l = line<KCONT>(i), q = quad<KCONT>(i);
            if constexpr (KCONT) {
                const int m = l ^ (4 * q);
                s.g[buf][4 * q][m] = v[i].x;
                s.g[buf][4 * q + 1][m] = v[i].y;
                s.g[buf][4 * q + 2][m] = v[i].z;
                s.g[buf][4 * q + 3][m] = v[i].w;
            } else {
                *reinterpret_cast<float4 *>(&s.g[buf][l][4 * (q ^ ((l >> 2) & 7))]) = v[i];
            }
        }
    }
    // B's slice, NT / 32 float4s a thread: with n contiguous, line k, quad of n;
    // with k contiguous, line n, quad of k
    template <bool BK = false>
    static __device__ __forceinline__ int b_line(int i) {
        return (threadIdx.x + TG_THREADS * i) / (BK ? 8 : NT / 4);
    }
    template <bool BK = false>
    static __device__ __forceinline__ int b_quad(int i) {
        return (threadIdx.x + TG_THREADS * i) % (BK ? 8 : NT / 4);
    }
    template <bool BK>
    static __device__ __forceinline__ void put_b(Shared &s, int buf, const float4 (&v)[NT / 32]) {
#pragma unroll
        for (int i = 0; i < NT / 32; ++i) {
            const int l = b_line<BK>(i), q = b_quad<BK>(i);
            if constexpr (BK) {
                const int n = l ^ (4 * q);
                s.b[buf][4 * q][n] = v[i].x;
                s.b[buf][4 * q + 1][n] = v[i].y;
                s.b[buf][4 * q + 2][n] = v[i].z;
                s.b[buf][4 * q + 3][n] = v[i].w;
            } else {
                *reinterpret_cast<float4 *>(&s.b[buf][l][4 * (q ^ ((l >> 2) & 7))]) = v[i];
            }
        }
    }
    __device__ __forceinline__ void slice(const Shared &s, int buf) {
        const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll 8
        for (int k = 0; k < TG_K; ++k) {
            const int sw = (k >> 2) & 7;
            const float4 g0 = *reinterpret_cast<const float4 *>(&s.g[buf][k][4 * ((2 * ty) ^ sw)]);
            const float4 g1 = *reinterpret_cast<const float4 *>(&s.g[buf][k][4 * ((2 * ty + 1) ^ sw)]);
            const float2 g[4] = {make_float2(g0.x, g0.y), make_float2(g0.z, g0.w), make_float2(g1.x, g1.y),
                                 make_float2(g1.z, g1.w)};
            float b[TN];
            if constexpr (TN == 4) {
                const float4 t = *reinterpret_cast<const float4 *>(&s.b[buf][k][4 * (tx ^ sw)]);
                b[0] = t.x; b[1] = t.y; b[2] = t.z; b[3] = t.w;
            } else {
                const float2 t = *reinterpret_cast<const float2 *>(&s.b[buf][k][4 * ((tx >> 1) ^ sw) + 2 * (tx & 1)]);
                b[0] = t.x; b[1] = t.y;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int n = 0; n < TN; ++n) acc[i][n] = __ffma2_rn(g[i], make_float2(b[n], b[n]), acc[i][n]);
        }
    }
    // all slices 0 .. n - 1: load_g(slice, float4[4]) and load_b(slice, float4[NT / 32])
    template <bool KCONT, bool BK = false, class LG, class LB>
    __device__ __forceinline__ void run(Shared &s, int n, LG load_g, LB load_b) {
        float4 gv[4], bv[NT / 32];
        if (n > 0) {
            load_g(0, gv);
            load_b(0, bv);
        }
        __syncthreads();   // the last run's readers are done
        for (int i = 0; i < n; ++i) {
            put_g<KCONT>(s, i & 1, gv);
            put_b<BK>(s, i & 1, bv);
            __syncthreads();
            if (i + 1 < n) {
                load_g(i + 1, gv);
                load_b(i + 1, bv);
            }
            slice(s, i & 1);
        }
    }
    // output row 8 (threadIdx.x / 16) + r, column TN (threadIdx.x % 16) + n of the tile
    __device__ __forceinline__ float out(int r, int n) const { return r & 1 ? acc[r >> 1][n].y : acc[r >> 1][n].x; }
};

}  // namespace sigk
