// What a fit derives from the inverse factor, in one cooperatively launched kernel:
//   alpha = W^T (W y)                     FP64 and FP32
//   |W|_2, times 1.5                      twelve power iterations on W^T W (the engines' error estimates)
//   W rounded to FP32, max |W|            for the scoring engines' operands
// A GP is served by a team of blocks that meet at a barrier of their own.  A pass u = W v, v' = W^T u reads W twice: rows
// by warps (dealt to and fro, so that every warp gets the same length), then columns by blocks, 16 at a time.
// The weights ride on the first pass.  Vectors sit in shared memory; the norm of a new vector divides the next product, so
// that normalising costs no barrier.
//
// Bound: W from L2, 26 times 4 n^2 bytes, and 25 barriers.  Up to 160 observations one block per GP keeps W in shared
// memory instead and needs no barriers but its own (64 observations: 118 us by teams, 17 us by one block).  Before, 57
// launches of three kernels per pass: 0.90 ms for one GP of 4096 observations (now 0.31 ms), 0.12 ms and 0.2 ms of launches
// for one of 64.
#include <algorithm>

#include "r3_f64.cuh"
#include "r3_internal.cuh"

namespace r3 {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kCols = 16;   // columns of W a block sums at a time: 128 contiguous bytes per row

struct WeightArgs {
    const double* W;       // [batch][npad][npad]
    const float* y;        // [batch][n]
    int batch, n, npad, team, iters;   // iters = 0: weights only
    double* alpha64;       // [batch][npad]
    float* alpha32;        // [batch][npad]
    float* W32;            // [batch][npad][npad] or nullptr
    double* wnorm;         // [batch] or nullptr (iters = 0)
    unsigned* wmax;        // [batch] bit pattern of max |W|, zero on entry, or nullptr
    double *u, *v;         // [batch][2][npad], [batch][npad]
    double* npart;         // [batch][npad / 16] sums of squares of the new vector
    unsigned* barrier;     // [batch]
    int* status;
};

// u_i = W_i . v / nrm (and W_i . y) for the rows of this warp
template <bool V, bool Y>
__device__ __forceinline__ void rows_pass(const WeightArgs& a, int g, int warp_id, int nwarps, const double* v, double inv_nrm)
{
    const int lane = threadIdx.x % 32, n = a.n, npad = a.npad;
    const double* Wg = a.W + (size_t)g * npad * npad;
    const float* y = a.y + (size_t)g * n;
    double* u = a.u + (size_t)g * 2 * npad;
    float top = 0.f;
    // slots 0 .. npad-1 are the rows from the longest to the shortest; a warp walks them to and fro, so that all warps get
    // about the same length
    for (int turn = 0; turn * nwarps < npad; ++turn) {
        const int slot = turn * nwarps + ((turn & 1) ? nwarps - 1 - warp_id : warp_id);
        if (slot >= npad) continue;
        const int i = npad - 1 - slot;
        const double* Wr = Wg + (size_t)i * npad;
        double s0 = 0.0, s1 = 0.0, t0 = 0.0, t1 = 0.0;
        if (i < n) {
#pragma unroll 8
            for (int k = 2 * lane; k <= i; k += 64) {   // the entry right of the diagonal is a stored zero
                const double2 w = __ldcg(reinterpret_cast<const double2*>(Wr + k));
                if (V) {
                    const double2 x = *reinterpret_cast<const double2*>(v + k);
                    s0 = fma(w.x, x.x, s0);
                    s1 = fma(w.y, x.y, s1);
                }
                if (Y) {
                    t0 = fma(w.x, (double)__ldg(y + k), t0);
                    t1 = fma(w.y, k + 1 < n ? (double)__ldg(y + k + 1) : 0.0, t1);
                    if (a.wmax) top = fmaxf(top, fmaxf(fabsf((float)w.x), fabsf((float)w.y)));
                }
            }
        }
        if (Y && a.W32) {
            float* o = a.W32 + (size_t)g * npad * npad + (size_t)i * npad;
            for (int k = 2 * lane; k < npad; k += 64) {
                float2 f = make_float2(0.f, 0.f);
                if (k <= i) {
                    const double2 w = __ldcg(reinterpret_cast<const double2*>(Wr + k));
                    f = make_float2((float)w.x, (float)w.y);
                }
                *reinterpret_cast<float2*>(o + k) = f;
            }
        }
        double s = s0 + s1, t = t0 + t1;
        for (int o = 16; o > 0; o >>= 1) {
            if (V) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (Y) t += __shfl_xor_sync(0xffffffffu, t, o);
        }
        if (lane == 0) {
            if (V) u[i] = s * inv_nrm;
            if (Y) u[npad + i] = t;
        }
    }
    if (Y && a.wmax) {
        const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
        if (lane == 0 && m) atomicMax(&a.wmax[g], m);
    }
}

// v'_j = sum_{i >= j} W_ij u_i for 16 columns from j0 (and the weights)
template <bool V, bool Y>
__device__ __forceinline__ void columns_pass(const WeightArgs& a, int g, int j0, const double* u, const double* uy, double* red)
{
    const int t = threadIdx.x, w = t / 32, l = t % 32, npad = a.npad;
    const double* Wg = a.W + (size_t)g * npad * npad + j0 + 2 * (l % 8);
    double2 s = make_double2(0.0, 0.0), q = s;
#pragma unroll 8
    for (int i = j0 + w * 4 + l / 8; i < a.n; i += 4 * kWarps) {
        const double2 x = __ldcg(reinterpret_cast<const double2*>(Wg + (size_t)i * npad));
        if (V) {
            s.x = fma(x.x, u[i], s.x);
            s.y = fma(x.y, u[i], s.y);
        }
        if (Y) {
            q.x = fma(x.x, uy[i], q.x);
            q.y = fma(x.y, uy[i], q.y);
        }
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
        if (V) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (Y) {
            q.x += __shfl_xor_sync(0xffffffffu, q.x, o);
            q.y += __shfl_xor_sync(0xffffffffu, q.y, o);
        }
    }
    __syncthreads();   // red: [2][8 warps][16]
    if (l < 8) {
        if (V) *reinterpret_cast<double2*>(red + w * kCols + 2 * l) = s;
        if (Y) *reinterpret_cast<double2*>(red + (kWarps + w) * kCols + 2 * l) = q;
    }
    __syncthreads();
    if (t < 32) {
        const int c = t % kCols;
        const bool second = t >= kCols;
        double sum = 0.0;
        if (second ? Y : V)
            for (int ww = 0; ww < kWarps; ++ww) sum += red[((second ? kWarps : 0) + ww) * kCols + c];
        if (second && Y) {
            a.alpha64[(size_t)g * npad + j0 + c] = sum;
            a.alpha32[(size_t)g * npad + j0 + c] = (float)sum;
        }
        if (V) {
            if (!second) a.v[(size_t)g * npad + j0 + c] = sum;
            double sq = second ? 0.0 : sum * sum;
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (t == 0) a.npart[(size_t)g * (npad / kCols) + j0 / kCols] = sq;
        }
    }
}

// One block, W in shared memory: histories of at most kSmallRows observations.  A thread sums one part of one row (then of
// one column): the lanes of a warp take 32 neighbouring rows and the same entries of the vector, so that the matrix is read
// without bank conflicts (odd leading dimension) and the vector as broadcasts; the parts meet in shared memory.
constexpr int kSmallRows = 160;
constexpr int kSmallThreads = 1024;
constexpr int kSmallParts = 16;
__global__ void __launch_bounds__(kSmallThreads, 1) weights_small_kernel(const WeightArgs a)
{
    extern __shared__ __align__(16) double vec[];   // W [npad][npad + 1], x [npad], sums [parts][npad]
    __shared__ double part_norm[kSmallThreads / 32];
    const int t = threadIdx.x, lane = t % 32, warp = t / 32, npad = a.npad, n = a.n, ld = npad + 1;
    const int P = min(kSmallParts, kSmallThreads / npad), idx = t % npad, part = t / npad, block = idx & ~31;
    double *Ws = vec, *x = Ws + npad * ld, *sums = x + npad;
    // x <- sum of the parts times scale (zero beyond the history when asked for)
    auto gather = [&](double scale, bool zero_beyond) {
        __syncthreads();
        if (t < npad) {
            double s = 0.0;
            for (int p = 0; p < P; ++p) s += sums[p * npad + t];
            x[t] = zero_beyond && t >= n ? 0.0 : s * scale;
        }
        __syncthreads();
    };
    auto rows = [&]() {
        if (part < P) {
            double s[4] = {};
            const double* w = Ws + idx * ld;
            int k = part;
            for (; k + 3 * P < block + 32; k += 4 * P)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[e] = fma(w[k + e * P], x[k + e * P], s[e]);
            for (; k < block + 32; k += P) s[0] = fma(w[k], x[k], s[0]);
            sums[part * npad + idx] = (s[0] + s[1]) + (s[2] + s[3]);
        }
    };
    auto columns = [&]() {
        if (part < P) {
            double s[4] = {};
            const double* w = Ws + idx;
            int i = block + part;
            for (; i + 3 * P < npad; i += 4 * P)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[e] = fma(w[(i + e * P) * ld], x[i + e * P], s[e]);
            for (; i < npad; i += P) s[0] = fma(w[i * ld], x[i], s[0]);
            sums[part * npad + idx] = (s[0] + s[1]) + (s[2] + s[3]);
        }
    };
    auto norm = [&]() {
        double s = t < npad ? x[t] * x[t] : 0.0;
        if (warp < npad / 32) {
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) part_norm[warp] = s;
        }
        __syncthreads();
        double all = 0.0;
        for (int w = 0; w < npad / 32; ++w) all += part_norm[w];
        return sqrt(all);
    };
    for (int g = blockIdx.x; g < a.batch; g += gridDim.x) {
        const double* Wg = a.W + (size_t)g * npad * npad;
        float top = 0.f;
        __syncthreads();
#pragma unroll 4
        for (int i = warp; i < npad; i += kSmallThreads / 32)
            for (int k = lane; k < npad; k += 32) {
                const double w = Wg[i * npad + k];
                Ws[i * ld + k] = w;
                if (i < n) top = fmaxf(top, fabsf((float)w));
                if (a.W32) a.W32[((size_t)g * npad + i) * npad + k] = (float)w;
            }
        if (t < npad) x[t] = t < n ? (double)a.y[(size_t)g * n + t] : 0.0;
        if (a.wmax) {
            const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
            if (lane == 0 && m) atomicMax(&a.wmax[g], m);
        }
        __syncthreads();
        rows();
        gather(1.0, true);
        columns();
        gather(1.0, false);
        if (t < npad) {
            a.alpha64[(size_t)g * npad + t] = x[t];
            a.alpha32[(size_t)g * npad + t] = (float)x[t];
        }
        if (a.iters == 0) continue;
        __syncthreads();
        if (t < npad) x[t] = t < n ? 1.0 + 0.37 * ((t * 2654435761u >> 16) & 0xff) / 255.0 : 0.0;
        double nrm = norm();
        for (int it = 0; it < a.iters; ++it) {
            rows();
            gather(nrm > 0.0 ? 1.0 / nrm : 0.0, true);
            columns();
            gather(1.0, false);
            nrm = norm();
        }
        if (t == 0) a.wnorm[g] = 1.5 * sqrt(nrm);
    }
}

__global__ void __launch_bounds__(kThreads, 2) weights_kernel(const WeightArgs a)
{
    extern __shared__ __align__(16) double vec[];   // [2][npad]
    __shared__ __align__(16) double red[2 * kWarps * kCols];
    __shared__ double norm_s;
    const int t = threadIdx.x, npad = a.npad, n = a.n;
    const int rank = blockIdx.x % a.team, teams = gridDim.x / a.team;
    const int warp_id = rank * kWarps + t / 32, nwarps = a.team * kWarps;
    auto block_norm = [&](const double* x, int count, bool squares) {   // every block adds up the same numbers in the same order
        double s = 0.0;
        for (int i = t; i < count; i += kThreads) {
            const double e = squares ? __ldcg(x + i) : x[i] * x[i];
            s += e;
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        __syncthreads();
        if (t % 32 == 0) red[t / 32] = s;
        __syncthreads();
        if (t == 0) {
            double all = 0.0;
            for (int w = 0; w < kWarps; ++w) all += red[w];
            norm_s = sqrt(all);
        }
        __syncthreads();
        return norm_s;
    };
    for (int g = blockIdx.x / a.team; g < a.batch; g += teams) {
        unsigned target = 0;
        auto meet = [&]() {
            if (a.team == 1) {
                __syncthreads();
                return true;
            }
            return team_barrier(a.barrier + g, target, (unsigned)a.team, a.status);
        };
        auto stage = [&](const double* src, double* dst) {
            for (int i = 2 * t; i < npad; i += 2 * kThreads)
                *reinterpret_cast<double2*>(dst + i) = __ldcg(reinterpret_cast<const double2*>(src + i));
        };
        const double* ug = a.u + (size_t)g * 2 * npad;
        __syncthreads();
        double nrm = 1.0;
        if (a.iters > 0) {
            for (int i = t; i < npad; i += kThreads)
                vec[i] = i < n ? 1.0 + 0.37 * ((i * 2654435761u >> 16) & 0xff) / 255.0 : 0.0;
            __syncthreads();
            nrm = block_norm(vec, npad, false);
        }
        for (int it = 0; it < max(a.iters, 1); ++it) {
            const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
            if (it > 0) rows_pass<true, false>(a, g, warp_id, nwarps, vec, inv);
            else if (a.iters > 0) rows_pass<true, true>(a, g, warp_id, nwarps, vec, inv);
            else rows_pass<false, true>(a, g, warp_id, nwarps, vec, inv);
            if (!meet()) return;
            if (a.iters > 0) stage(ug, vec);
            if (it == 0) stage(ug + npad, vec + npad);
            __syncthreads();
            for (int c = rank; c < npad / kCols; c += a.team) {
                if (it > 0) columns_pass<true, false>(a, g, c * kCols, vec, vec, red);
                else if (a.iters > 0) columns_pass<true, true>(a, g, c * kCols, vec, vec + npad, red);
                else columns_pass<false, true>(a, g, c * kCols, vec, vec + npad, red);
            }
            if (a.iters == 0) break;
            if (!meet()) return;
            nrm = block_norm(a.npart + (size_t)g * (npad / kCols), npad / kCols, true);
            if (it + 1 < a.iters) {
                stage(a.v + (size_t)g * npad, vec);
                __syncthreads();
            }
        }
        // the last norm estimates |W|_2^2 from below; 1.5 covers slow convergence
        if (a.wnorm && rank == 0 && t == 0) a.wnorm[g] = 1.5 * sqrt(nrm);
    }
}

}  // namespace

size_t weights_scratch_doubles(int batch, int npad) { return (size_t)batch * (3 * (size_t)npad + npad / kCols); }

r3_status_t weights_device(const WeightProblem& p, double* scratch, unsigned* barrier, int* status, int device,
                           cudaStream_t stream)
{
    WeightArgs a;
    a.W = p.W; a.y = p.y;
    a.batch = p.batch; a.n = p.n; a.npad = p.npad;
    a.iters = p.wnorm ? 12 : 0;
    a.alpha64 = p.alpha64; a.alpha32 = p.alpha32; a.W32 = p.W32; a.wnorm = p.wnorm; a.wmax = p.wmax;
    a.u = scratch;
    a.v = a.u + (size_t)p.batch * 2 * p.npad;
    a.npart = a.v + (size_t)p.batch * p.npad;
    a.barrier = barrier;
    a.status = status;
    int sms = 148;
    R3_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    if (p.npad <= kSmallRows) {
        const size_t small = sizeof(double) * ((size_t)p.npad * (p.npad + 2) + std::min(kSmallParts * p.npad, kSmallThreads));
        a.team = 1;
        R3_CUDA_TRY(cudaFuncSetAttribute(weights_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sizeof(double) * (kSmallRows * (kSmallRows + 2) + kSmallThreads))));
        R3_LAUNCH(weights_small_kernel, std::min(p.batch, sms), kSmallThreads, small, stream, a);
        return R3_OK;
    }
    const size_t smem = sizeof(double) * 2 * p.npad;
    R3_CUDA_TRY(cudaFuncSetAttribute(weights_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(double) * 2 * kMaxN)));
    const int resident = sms * (smem <= 96 * 1024 ? 2 : 1);
    a.team = std::max(1, std::min(p.npad / kCols, resident / p.batch));   // one block per 16 columns as far as the GPU goes round
    const unsigned grid = (unsigned)(a.team * std::min(p.batch, resident / a.team));
    void* params[] = {&a};
    R3_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)weights_kernel, dim3(grid), dim3(kThreads), params, smem, stream));
    ++g_launches;
    return R3_OK;
}

}  // namespace r3
