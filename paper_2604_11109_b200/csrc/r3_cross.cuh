// FP64 pieces shared by the accuracy guard's rescue and the batch proposal: a tile of cross-covariances and a tile of a
// product with transposed second operand.  Blocks of 256 threads.
#pragma once

#include "r3_f64.cuh"
#include "r3_internal.cuh"

namespace r3 {

constexpr int kCrossThreads = 256;
constexpr int kCrossTile = 64;
constexpr int kCrossStages = 3;       // 16-deep operand stages in flight
constexpr size_t kCrossStageBytes = sizeof(double) * kCrossStages * 2 * kCrossTile * kStageLd;

// k(z_c, x_k) and the partial means of (CT rows z) x (64 rows x from column 64 kb), CT / 16 x 4 of them per thread.
// zrow(c), xrow(k): the raw rows (nullptr: a row of zeros, its values are not used; xrow is asked for k < n only).
// store(c, k, value) for every c < CT and every k < npad of the block (zero beyond n), mean(c, sum over the block of
// value * alpha) once per c unless alpha is nullptr.
template <int CT, class ZRow, class XRow, class Store, class Mean>
__device__ __forceinline__ void cross_tile(int n, int d, int npad, const float* ell, double sf2, const double* alpha, ZRow zrow,
                                           XRow xrow, int kb, unsigned char* smem, Store store, Mean mean)
{
    constexpr int U = CT / 16;
    float* zs = reinterpret_cast<float*>(smem);   // [CT][33]
    float* xs = zs + CT * 33;                     // [64][33]
    double* il = reinterpret_cast<double*>(xs + 64 * 33 + (CT * 33) % 2);   // [32] reciprocal lengthscales
    const float** zp = reinterpret_cast<const float**>(il + 32);            // [CT] rows of the tile
    const float** xp = zp + CT;                                             // [64]
    const int t = threadIdx.x, tx = t % 16, ty = t / 16;
    const int k0 = kb * 64;
    double r2[U][4] = {};
    __syncthreads();
    if (t < CT) zp[t] = zrow(t);
    else if (t >= 128 && t < 192) xp[t - 128] = k0 + t - 128 < n ? xrow(k0 + t - 128) : nullptr;
    for (int c0 = 0; c0 < d; c0 += 32) {
        __syncthreads();
        // all of a thread's loads are under way before the first is stored
        const int c = t % 32, r0 = t / 32;
        float zv[CT / 8], xv[8];
#pragma unroll
        for (int e = 0; e < CT / 8; ++e) {
            const float* p = zp[r0 + 8 * e];
            zv[e] = (p && c0 + c < d) ? p[c0 + c] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float* p = xp[r0 + 8 * e];
            xv[e] = (p && c0 + c < d) ? p[c0 + c] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < CT / 8; ++e) zs[(r0 + 8 * e) * 33 + c] = zv[e];
#pragma unroll
        for (int e = 0; e < 8; ++e) xs[(r0 + 8 * e) * 33 + c] = xv[e];
        if (t < 32) il[t] = (c0 + t < d) ? 1.0 / (double)ell[c0 + t] : 0.0;
        __syncthreads();
        const int cmax = min(32, d - c0);
        for (int c = 0; c < cmax; ++c) {
            double z[U], x[4];
#pragma unroll
            for (int u = 0; u < U; ++u) z[u] = (double)zs[(ty + 16 * u) * 33 + c];
#pragma unroll
            for (int v = 0; v < 4; ++v) x[v] = (double)xs[(tx + 16 * v) * 33 + c];
            const double w = il[c];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const double df = (x[v] - z[u]) * w;
                    r2[u][v] = fma(df, df, r2[u][v]);
                }
        }
    }
#pragma unroll 1
    for (int u = 0; u < U; ++u) {   // not unrolled: four square roots and exponentials at a time are enough to overlap
        double part = 0.0, ru[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            ru[v] = r2[0][v];
#pragma unroll
            for (int uu = 1; uu < U; ++uu) ru[v] = uu == u ? r2[uu][v] : ru[v];
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int k = k0 + tx + 16 * v;
            if (k >= npad) continue;
            double kv = 0.0;
            if (k < n) {
                const double sq = sqrt(5.0) * sqrt(ru[v]);
                kv = sf2 * fma(sq, fma(sq, 1.0 / 3.0, 1.0), 1.0) * exp(-sq);
                if (alpha) part = fma(kv, alpha[k], part);
            }
            store(ty + 16 * u, k, kv);
        }
        if (alpha) {
            for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            if (tx == 0) mean(ty + 16 * u, part);
        }
    }
}

// c += A B^T for 64 rows of A and of B (row-major, leading dimension ld, rows from arows / brows on are zeros), columns
// [0, K), K a multiple of 16: warp w holds rows 16 (w % 4) + 8 i + l / 4 and columns 32 (w / 4) + 8 j + 2 (l % 4) + h.
__device__ __forceinline__ void nt_tile(const double* A, int arows, const double* B, int brows, int ld, int K,
                                        unsigned char* smem, double (&c)[2][4][2], int* status)
{
    double* sA = reinterpret_cast<double*>(smem);         // [stages][64][20]
    double* sB = sA + kCrossStages * kCrossTile * kStageLd;
    const int t = threadIdx.x, w = t / 32, l = t % 32;
    const int wm = (w % 4) * 16, wn = (w / 4) * 32;
    const int steps = K / 16;
    auto load = [&](int s, int k0) {
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            const int e = t + kCrossThreads * it, r = e / 8, q = e % 8;
            cp_async16(sA + (s * kCrossTile + r) * kStageLd + 2 * q, A + (size_t)(r < arows ? r : 0) * ld + R3_IDX(k0 + 2 * q, ld - 1, status), r < arows);
            cp_async16(sB + (s * kCrossTile + r) * kStageLd + 2 * q, B + (size_t)(r < brows ? r : 0) * ld + R3_IDX(k0 + 2 * q, ld - 1, status), r < brows);
        }
    };
    __syncthreads();   // earlier reads of the stages' bytes are done
#pragma unroll
    for (int s = 0; s < kCrossStages - 1; ++s) {
        if (s < steps) load(s, s * 16);
        cp_async_commit();
    }
    for (int kb = 0; kb < steps; ++kb) {
        cp_async_wait<kCrossStages - 2>();
        __syncthreads();
        if (kb + kCrossStages - 1 < steps) load((kb + kCrossStages - 1) % kCrossStages, (kb + kCrossStages - 1) * 16);
        cp_async_commit();
        const double* pa = sA + ((kb % kCrossStages) * kCrossTile + wm + l / 4) * kStageLd + l % 4;
        const double* pb = sB + ((kb % kCrossStages) * kCrossTile + wn + l / 4) * kStageLd + l % 4;
#pragma unroll
        for (int kk = 0; kk < 16; kk += 4) {
            double fa[2], fb[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) fa[i] = pa[i * 8 * kStageLd + kk];
#pragma unroll
            for (int j = 0; j < 4; ++j) fb[j] = pb[j * 8 * kStageLd + kk];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dmma(c[i][j], fa[i], fb[j]);
        }
    }
    cp_async_wait<0>();
    __syncthreads();
}

}  // namespace r3
