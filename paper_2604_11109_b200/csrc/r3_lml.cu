// Log marginal likelihood of the history and its gradient with respect to the logarithms of the
// hyper-parameters, from what the fit already holds (L, W = L^-1, alpha, X, y):
//     lml = -1/2 y.alpha - sum_i log L_ii - n/2 log(2 pi)
//     M   = alpha alpha^T - K^-1,   K^-1 = W^T W
//     d lml / d log ell_j = 1/2 sum_ik M_ik sf2 e^-s (5/3)(1 + s) u_j^2     (u_j = (x_ij - x_kj)/ell_j)
//     d lml / d log sf2   = 1/2 sum_ik M_ik Kf_ik,    d lml / d log sn2 = 1/2 sn2 trace(M)
// Everything in FP64.  A block forms a 64 x 64 tile of the lower triangle of K^-1 on the FP64 tensor path and, with the
// tile still in registers, its share of every pair sum; M is never stored.  The sums are reduced in a fixed order (per-tile
// partial sums, then one warp per derivative adds them), so results repeat bit for bit.
// Bound: FP64 rate, n^3/3 multiply-adds for K^-1 and 6 n^2 d / 2 operations for the pairs (a feature's scale is applied to
// its sum, not to every pair).  64 GPs of 512 observations, 32 features: 0.34 ms; K^-1 by 4x4 register tiles, M written and
// read back, and a warp sum per feature and pair tile: 0.79 ms.
#include <math.h>

#include <algorithm>
#include <vector>

#include "r3_f64.cuh"
#include "r3_internal.cuh"

namespace r3 {

namespace {

constexpr int kThreads = 256;
constexpr int kTile = 64;
constexpr int kStages = 3;
constexpr int kLd = 68;   // leading dimension of a [16][64] operand stage: 4 mod 16 keeps the fragment reads on different banks
constexpr size_t kTileSmem = sizeof(double) * kStages * 2 * 16 * kLd;   // 52 KB; the pair sums need 34 KB of it

struct LmlArgs {
    const float *X, *ell, *sf2, *sn2, *y;
    const double *W, *L, *alpha;
    int n, d, npad, tiles;
    double* partial;   // [batch][tiles][d + 2]: the features' sums, sum w M Kf, trace
    double* out;       // [batch][d + 3]
    int* status;       // status words, for the index checks of the bounds-checking build
};

__global__ void __launch_bounds__(kThreads, 2) lml_tile_kernel(const LmlArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[8][34];   // the warps' sums of 32 features, of M Kf and of the trace
    const int g = blockIdx.y, n = a.n, d = a.d, npad = a.npad;
    const int t = threadIdx.x, w = t / 32, l = t % 32, wm = (w % 4) * 16, wn = (w / 4) * 32;
    // tile index -> (ti, tj) of the lower triangle; small ti have the longest reductions and come first
    int ti = (int)((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);
    while ((ti + 1) * (ti + 2) / 2 <= (int)blockIdx.x) ++ti;
    while (ti * (ti + 1) / 2 > (int)blockIdx.x) --ti;
    const int tj = blockIdx.x - ti * (ti + 1) / 2, i0 = ti * kTile, j0 = tj * kTile;
    const double* Wg = a.W + (size_t)g * npad * npad;
    // ---- c = sum_{r >= i0} W[r][i] W[r][j]
    double c[2][4][2] = {};
    {
        double* sA = reinterpret_cast<double*>(smem);   // [stages][16][68]
        double* sB = sA + kStages * 16 * kLd;
        const int steps = (npad - i0) / 16;             // npad and i0 are multiples of 32
        auto load = [&](int s, int r0) {
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                const int e = t + kThreads * it, r = e / 32, q = e % 32;
                // the last tile of a row or column may have 32 columns only
                const bool oki = i0 + 2 * q < npad, okj = j0 + 2 * q < npad;
                const size_t row = (size_t)R3_IDX(r0 + r, npad, a.status) * npad;
                cp_async16(sA + (s * 16 + r) * kLd + 2 * q, Wg + row + R3_IDX(oki ? i0 + 2 * q : 0, npad - 1, a.status), oki);
                cp_async16(sB + (s * 16 + r) * kLd + 2 * q, Wg + row + R3_IDX(okj ? j0 + 2 * q : 0, npad - 1, a.status), okj);
            }
        };
#pragma unroll
        for (int s = 0; s < kStages - 1; ++s) {
            if (s < steps) load(s, i0 + s * 16);
            cp_async_commit();
        }
        for (int s = 0; s < steps; ++s) {
            cp_async_wait<kStages - 2>();
            __syncthreads();
            if (s + kStages - 1 < steps) load((s + kStages - 1) % kStages, i0 + (s + kStages - 1) * 16);
            cp_async_commit();
            const double* pa = sA + ((s % kStages) * 16 + l % 4) * kLd + wm + l / 4;
            const double* pb = sB + ((s % kStages) * 16 + l % 4) * kLd + wn + l / 4;
#pragma unroll
            for (int kk = 0; kk < 16; kk += 4) {
                double fa[2], fb[4];
#pragma unroll
                for (int i = 0; i < 2; ++i) fa[i] = pa[kk * kLd + 8 * i];
#pragma unroll
                for (int j = 0; j < 4; ++j) fb[j] = pb[kk * kLd + 8 * j];
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) dmma(c[i][j], fa[i], fb[j]);
            }
        }
        cp_async_wait<0>();
    }
    // ---- the pairs: rows wm + 8 i + l / 4, columns wn + 8 j + 2 (l % 4) + h of the tile
    double* xi = reinterpret_cast<double*>(smem);   // [64][33]
    double* xj = xi + kTile * 33;
    double* il = xj + kTile * 33;                   // [32] reciprocal lengthscales (FP64, as the fit's)
    const float* Xg = a.X + (size_t)g * n * d;
    auto stage = [&](int c0) {
        __syncthreads();
        const int f = t % 32, q = t / 32;
        float vi[8], vj[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int gi = i0 + q + 8 * e, gj = j0 + q + 8 * e;
            vi[e] = (gi < n && c0 + f < d) ? __ldg(Xg + R3_IDX((size_t)gi * d + c0 + f, (size_t)n * d, a.status)) : 0.f;
            vj[e] = (gj < n && c0 + f < d) ? __ldg(Xg + R3_IDX((size_t)gj * d + c0 + f, (size_t)n * d, a.status)) : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            xi[(q + 8 * e) * 33 + f] = (double)vi[e];
            xj[(q + 8 * e) * 33 + f] = (double)vj[e];
        }
        if (t < 32) il[t] = (c0 + t < d) ? 1.0 / (double)a.ell[(size_t)g * d + c0 + t] : 0.0;
        __syncthreads();
    };
    double r2[2][4][2] = {};
    for (int c0 = 0; c0 < d; c0 += 32) {
        stage(c0);
        const int cmax = min(32, d - c0);
        for (int f = 0; f < cmax; ++f) {
            const double s = il[f];
            double p[2], q[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) p[i] = xi[(wm + 8 * i + l / 4) * 33 + f];
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) q[j][h] = xj[(wn + 8 * j + 2 * (l % 4) + h) * 33 + f];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const double df = (p[i] - q[j][h]) * s;
                        r2[i][j][h] = fma(df, df, r2[i][j][h]);
                    }
        }
    }
    // c becomes the weight of u^2 in the lengthscales' derivatives: w M sf2 e^-s (5/3)(1 + s)
    const double sf2 = (double)a.sf2[g];
    const double* alpha = a.alpha + (size_t)g * npad;
    double kf = 0.0, trace = 0.0;
#pragma unroll 1
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = i0 + wm + 8 * i + l / 4, col = j0 + wn + 8 * j + 2 * (l % 4) + h;
                double r = 0.0, k = 0.0;   // j is not unrolled (code size): pick its entries
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    r = jj == j ? r2[i][jj][h] : r;
                    k = jj == j ? c[i][jj][h] : k;
                }
                double gk = 0.0;
                if (row < n && col <= row) {
                    const double m = fma(alpha[row], alpha[col], -k), wm2 = row == col ? m : 2.0 * m;
                    const double s = sqrt(5.0) * sqrt(r), e = wm2 * sf2 * exp(-s);
                    gk = e * (5.0 / 3.0) * (1.0 + s);
                    kf = fma(e, fma(s, fma(s, 1.0 / 3.0, 1.0), 1.0), kf);
                    if (row == col) trace += m;
                }
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) c[i][jj][h] = jj == j ? gk : c[i][jj][h];
            }
    double* out = a.partial + ((size_t)g * a.tiles + blockIdx.x) * (d + 2);
    auto warp_sum = [](double v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    kf = warp_sum(kf);
    trace = warp_sum(trace);
    if (l == 0) {
        red[w][32] = kf;
        red[w][33] = trace;
    }
    for (int c0 = 0; c0 < d; c0 += 32) {
        if (d > 32) stage(c0);   // with one chunk the coordinates are still there
        const int cmax = min(32, d - c0);
        // Eight features at a time: every lane has eight sums, and a butterfly that halves their number with the number of
        // lanes that hold them needs 9 exchanges instead of 40.
#pragma unroll 1
        for (int f0 = 0; f0 < cmax; f0 += 8) {
            double v[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const int f = f0 + b;   // beyond cmax: coordinates and scale are zeros
                const double s = il[f];
                double acc = 0.0, q[4][2];
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int h = 0; h < 2; ++h) q[j][h] = xj[(wn + 8 * j + 2 * (l % 4) + h) * 33 + f];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const double p = xi[(wm + 8 * i + l / 4) * 33 + f];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const double u = p - q[j][h];
                            acc = fma(c[i][j][h] * u, u, acc);
                        }
                }
                v[b] = acc * (s * s);   // the scale of u_j^2, once per sum
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                const bool up = (l & o) != 0;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (b < o) {
                        const double give = up ? v[b] : v[b + o], keep = up ? v[b + o] : v[b];
                        v[b] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
            }
            double s = v[0];   // of feature f0 + l % 8
            s += __shfl_xor_sync(0xffffffffu, s, 8);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            if (l < 8) red[w][f0 + l] = s;
        }
        __syncthreads();
        if (t < cmax || (c0 == 0 && t >= 32 && t < 34)) {
            double s = 0.0;
            for (int ww = 0; ww < 8; ++ww) s += red[ww][t];
            out[R3_IDX(t < 32 ? c0 + t : d + t - 32, d + 2, a.status)] = s;
        }
        __syncthreads();
    }
}

// A warp per derivative (and one each for the trace and the value), the tiles' sums added in a fixed order.
__global__ void __launch_bounds__(kThreads) lml_finish_kernel(const LmlArgs a)
{
    const int g = blockIdx.y, lane = threadIdx.x % 32, what = blockIdx.x * (kThreads / 32) + threadIdx.x / 32, d = a.d, n = a.n;
    if (what > d + 2) return;
    double* out = a.out + (size_t)g * (d + 3);
    double s = 0.0;
    if (what <= d + 1) {
        const double* p = a.partial + (size_t)g * a.tiles * (d + 2) + what;
#pragma unroll 4
        for (int b = lane; b < a.tiles; b += 32) s += p[(size_t)b * (d + 2)];
    } else {
        const double* L = a.L + (size_t)g * a.npad * a.npad;
#pragma unroll 4
        for (int i = lane; i < n; i += 32) {
            s = fma(-0.5 * (double)a.y[(size_t)g * n + i], a.alpha[(size_t)g * a.npad + i], s);
            s -= log(L[(size_t)i * a.npad + i]);
        }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        if (what <= d) out[1 + what] = 0.5 * s;
        else if (what == d + 1) out[d + 2] = 0.5 * (double)a.sn2[g] * s;
        else out[0] = s - 0.5 * n * 1.8378770664093454836;   // log(2 pi)
    }
}

int lml_tiles(int n) { return ((n + kTile - 1) / kTile) * ((n + kTile - 1) / kTile + 1) / 2; }

}  // namespace

size_t lml_scratch_doubles(const r3_fit_state& s) { return (size_t)s.batch * ((size_t)lml_tiles(s.n) * (s.d + 2) + s.d + 3); }

// Asynchronous: *out (device, inside scratch) becomes [batch][d + 3] = {lml, d/dlog ell_1..d, d/dlog sf2, d/dlog sn2}.
r3_status_t lml_enqueue(const r3_fit_state& s, double* scratch, double** out, int* status, cudaStream_t stream)
{
    LmlArgs a;
    a.status = status;
    a.X = s.X; a.ell = s.ell_d; a.sf2 = s.sf2_d; a.sn2 = s.sn2_d; a.y = s.y;
    a.W = s.W64; a.L = s.L64; a.alpha = s.alpha64;
    a.n = s.n; a.d = s.d; a.npad = s.npad;
    a.tiles = lml_tiles(s.n);
    a.out = scratch;
    a.partial = scratch + (size_t)s.batch * (s.d + 3);
    *out = a.out;
    R3_CUDA_TRY(cudaFuncSetAttribute(lml_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem));
    R3_LAUNCH(lml_tile_kernel, dim3(a.tiles, s.batch), kThreads, kTileSmem, stream, a);
    R3_LAUNCH(lml_finish_kernel, dim3((s.d + 3 + kThreads / 32 - 1) / (kThreads / 32), s.batch), kThreads, 0, stream, a);
    return R3_OK;
}

// out_h: host [batch][d + 3].  Synchronises.
r3_status_t lml_device(r3_gp* gp, double* out_h, cudaStream_t stream)
{
    double* scratch = nullptr;
    auto done = [&](r3_status_t st) {
        if (st != R3_OK) cudaStreamSynchronize(stream);   // otherwise it has been
        FreeScope no_wait;
        dev_free(scratch);
        return st;
    };
    R3_CUDA_TRY(dev_malloc(&scratch, sizeof(double) * lml_scratch_doubles(*gp)));
    double* out = nullptr;
    const r3_status_t st = lml_enqueue(*gp, scratch, &out, gp->status_d, stream);
    if (st != R3_OK) return done(st);
    cudaError_t e = cudaMemcpyAsync(out_h, out, sizeof(double) * (size_t)gp->batch * (gp->d + 3), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        set_error("r3_gp_lml: %s", cudaGetErrorString(e));
        return done(R3_ERR_CUDA);
    }
    return done(R3_OK);
}

}  // namespace r3
