// r3_gp_fit and r3_gp_append on the device: factor and inverse factor (r3_factor.cu), weights, norm estimate.
//
// Everything here runs once per BO round, in FP64, and is rounded to FP32 once at the end:
//   K = L L^T, W = L^-1          factor_device
//   alpha = W^T (W y)            two triangular matrix-vector products
//   |W|_2                        power iteration, for the scoring engines' error estimates
// `batch` GPs go together.  n is padded to a multiple of 32 with an identity block, which leaves L, W and alpha unchanged.
#include "r3_internal.cuh"

namespace r3 {

namespace {

// ------------------------------------------------------------------------------------ weights
// u = W y (lower-triangular W, one warp per row); rows >= n give 0.
template <typename T>
__global__ void w_times_y_kernel(const double* __restrict__ W, const T* __restrict__ y, int ystride, int n,
                                 int npad, double* __restrict__ u)
{
    const int g = blockIdx.y;
    const int row = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    if (row >= npad) return;
    const double* Wr = W + (size_t)g * npad * npad + (size_t)row * npad;
    double s = 0.0;
    if (row < n)
        for (int k = lane; k <= row; k += 32) s += Wr[k] * (double)y[(size_t)g * ystride + k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) u[(size_t)g * npad + row] = s;
}

// alpha = W^T u in two steps so that n = 4096 still fills the GPU: the rows are cut into kRowSlabs
// slabs, each block sums one slab for 128 columns (coalesced across columns), then the slabs are added
// in a fixed order (deterministic).
constexpr int kRowSlabs = 32;
__global__ void wt_times_u_partial_kernel(const double* __restrict__ W, const double* __restrict__ u, int n,
                                          int npad, double* __restrict__ partial)
{
    const int g = blockIdx.z, slab = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= npad) return;
    const int rows = (npad + kRowSlabs - 1) / kRowSlabs;
    const int i0 = max(slab * rows, j), i1 = min(min((slab + 1) * rows, npad), n);
    const double* Wg = W + (size_t)g * npad * npad;
    double s = 0.0;
    if (j < n)
        for (int i = i0; i < i1; ++i) s += Wg[(size_t)i * npad + j] * u[(size_t)g * npad + i];
    partial[((size_t)g * kRowSlabs + slab) * npad + j] = s;
}

__global__ void wt_times_u_reduce_kernel(const double* __restrict__ partial, int npad,
                                         double* __restrict__ alpha64, float* __restrict__ alpha32)
{
    const int g = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= npad) return;
    double s = 0.0;
    for (int r = 0; r < kRowSlabs; ++r) s += partial[((size_t)g * kRowSlabs + r) * npad + j];
    alpha64[(size_t)g * npad + j] = s;
    alpha32[(size_t)g * npad + j] = (float)s;
}

// Power iteration on W^T W: v holds the current vector (unit norm after the call), lam its norm
// before normalisation, i.e. the current estimate of |W|_2^2.
__global__ void power_init_kernel(double* __restrict__ v, int n, int npad)
{
    const int g = blockIdx.x;
    for (int i = threadIdx.x; i < npad; i += blockDim.x)
        v[(size_t)g * npad + i] = (i < n) ? (1.0 + 0.37 * ((i * 2654435761u >> 16) & 0xff) / 255.0) : 0.0;
}

__global__ void power_normalize_kernel(double* __restrict__ v, int npad, double* __restrict__ lam)
{
    __shared__ double s[256];
    const int g = blockIdx.x;
    double* vg = v + (size_t)g * npad;
    double acc = 0.0;
    for (int i = threadIdx.x; i < npad; i += 256) acc += vg[i] * vg[i];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    const double nrm = sqrt(s[0]);
    if (threadIdx.x == 0) lam[g] = nrm;
    const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
    for (int i = threadIdx.x; i < npad; i += 256) vg[i] *= inv;
}

__global__ void power_finish_kernel(const double* __restrict__ lam, double* __restrict__ wnorm, int batch)
{
    // lam ~ |W|_2^2 from below; 1.5 covers slow convergence
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < batch) wnorm[g] = 1.5 * sqrt(lam[g]);
}

__global__ void to_float_kernel(const double* __restrict__ a, float* __restrict__ b, size_t count)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count;
         i += (size_t)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

// From W and y: the estimate of |W|_2 (power iteration on W^T W; alpha64/alpha32 serve as scratch first),
// alpha = W^T (W y) in FP64 and FP32, and W rounded to FP32.  u: [B][npad] scratch; slabs: [B + B*kRowSlabs*npad].
r3_status_t finish_weights(int B, int n, int npad, const double* W64, const float* y, double* alpha64, float* alpha32,
                           float* W32, double* wnorm_d, double* u, double* slabs, cudaStream_t stream)
{
    double* pv = alpha64;
    double* lam = slabs;  // [B], followed by the row-slab partial sums
    double* part = slabs + B;
    R3_LAUNCH(power_init_kernel, B, 256, 0, stream, pv, n, npad);
    R3_LAUNCH(power_normalize_kernel, B, 256, 0, stream, pv, npad, lam);
    for (int it = 0; it < 12; ++it) {
        R3_LAUNCH(w_times_y_kernel<double>, dim3((npad + 7) / 8, B), 256, 0, stream, W64, pv, npad, n, npad, u);
        R3_LAUNCH(wt_times_u_partial_kernel, dim3((npad + 127) / 128, kRowSlabs, B), 128, 0, stream, W64, u, n, npad,
                  part);
        R3_LAUNCH(wt_times_u_reduce_kernel, dim3((npad + 127) / 128, B), 128, 0, stream, part, npad, pv, alpha32);
        R3_LAUNCH(power_normalize_kernel, B, 256, 0, stream, pv, npad, lam);
    }
    R3_LAUNCH(power_finish_kernel, (B + 255) / 256, 256, 0, stream, lam, wnorm_d, B);
    R3_LAUNCH(w_times_y_kernel<float>, dim3((npad + 7) / 8, B), 256, 0, stream, W64, y, n, n, npad, u);
    R3_LAUNCH(wt_times_u_partial_kernel, dim3((npad + 127) / 128, kRowSlabs, B), 128, 0, stream, W64, u, n, npad, part);
    R3_LAUNCH(wt_times_u_reduce_kernel, dim3((npad + 127) / 128, B), 128, 0, stream, part, npad, alpha64, alpha32);
    R3_LAUNCH(to_float_kernel, 1184, 256, 0, stream, W64, W32, (size_t)B * npad * npad);
    return R3_OK;
}

}  // namespace

// Runs the whole fit on `stream`.  gp->X, ell (device copies) and the scalar arrays are already in
// place; L64, W64, W32, alpha*, best_d are filled.  The caller synchronises and reads status_d.
r3_status_t fit_device(r3_gp* gp, const float* y, cudaStream_t stream)
{
    const int B = gp->batch, npad = gp->npad;
    double *u = nullptr, *slabs = nullptr;
    void* scratch = nullptr;
    auto done = [&](r3_status_t st) {
        dev_free(u);
        dev_free(slabs);
        dev_free(scratch);
        return st;
    };
#define TRY_DONE(expr)                                                                             \
    do {                                                                                           \
        cudaError_t e__ = (expr);                                                                  \
        if (e__ != cudaSuccess) {                                                                  \
            set_error("%s failed: %s", #expr, cudaGetErrorString(e__));                            \
            return done(e__ == cudaErrorMemoryAllocation ? R3_ERR_ALLOC : R3_ERR_CUDA);            \
        }                                                                                          \
    } while (0)
    TRY_DONE(dev_malloc(&u, sizeof(double) * B * npad));
    TRY_DONE(dev_malloc(&slabs, sizeof(double) * ((size_t)B + (size_t)B * kRowSlabs * npad)));
    TRY_DONE(dev_malloc(&scratch, factor_scratch_bytes(B, npad)));
    FactorProblem f;
    f.X = gp->X; f.y = y; f.ell = gp->ell_d; f.sf2 = gp->sf2_d; f.sn2 = gp->sn2_d;
    f.batch = B; f.n = gp->n; f.d = gp->d; f.npad = npad; f.rows_done = 0;
    f.L = gp->L64; f.W = gp->W64;
    f.best = gp->best_d; f.yabs = gp->yabs_d;
    r3_status_t st = factor_device(f, scratch, gp->status_d, gp->device, stream);
    if (st != R3_OK) return done(st);
    st = finish_weights(B, gp->n, npad, gp->W64, y, gp->alpha64, gp->alpha32, gp->W32, gp->wnorm_d, u, slabs, stream);
    if (st != R3_OK) return done(st);
    TRY_DONE(cudaMemcpyAsync(gp->status_h, gp->status_d, 2 * sizeof(int), cudaMemcpyDeviceToHost, stream));
    TRY_DONE(cudaStreamSynchronize(stream));
#undef TRY_DONE
    return done(R3_OK);  // frees the temporaries
}

// =====================================================================================================
// r3_gp_append: k more observations per GP without refactoring what is already factored.  The rows of L and W of whole
// tiles of old observations are copied, the rows below are computed as a fit computes them (r3_factor.cu): O(k n^2)
// against the fit's O(n^3 / 3), and the result is the one a fit of the concatenated history gives.
namespace {

// Rows [0, rows) of L and W of every GP into matrices with another leading dimension (the columns right of the copied
// triangle are zeroed by the factorisation, or lie within the copied width and are zero there).
__global__ void embed_kernel(const double* __restrict__ L0, const double* __restrict__ W0, int np0, double* __restrict__ L1,
                             double* __restrict__ W1, int np1, int rows)
{
    const int g = blockIdx.y, i = blockIdx.x;
    const double* src = (blockIdx.z ? W0 : L0) + (size_t)g * np0 * np0 + (size_t)i * np0;
    double* dst = (blockIdx.z ? W1 : L1) + (size_t)g * np1 * np1 + (size_t)i * np1;
    for (int c = 2 * threadIdx.x; c < rows; c += 2 * blockDim.x)
        *reinterpret_cast<double2*>(dst + c) = *reinterpret_cast<const double2*>(src + c);
}

struct AppendBuffers {
    float *X = nullptr, *y = nullptr, *W32 = nullptr, *alpha32 = nullptr, *best = nullptr;   // best: [2][B]
    double *L64 = nullptr, *W64 = nullptr, *alpha64 = nullptr, *u = nullptr, *slabs = nullptr, *wnorm = nullptr;
    void* scratch = nullptr;
    void release()
    {
        dev_free(X); dev_free(y); dev_free(W32); dev_free(alpha32); dev_free(L64); dev_free(W64); dev_free(alpha64);
        dev_free(u); dev_free(slabs); dev_free(best); dev_free(wnorm); dev_free(scratch);
        *this = AppendBuffers();
    }
};

}  // namespace

r3_status_t append_device(r3_gp* gp, const float* Xnew, const float* ynew, int k, cudaStream_t stream)
{
    const size_t xnew_gp_stride = (size_t)k * gp->d, ynew_gp_stride = (size_t)k;
    const int B = gp->batch, d = gp->d, n0 = gp->n, n1 = n0 + k, np0 = gp->npad, np1 = round_up(n1, kFitBlock);
    const size_t mat1 = (size_t)np1 * np1;
    AppendBuffers nb;
    auto fail = [&](r3_status_t st) {
        nb.release();
        return st;
    };
#define TRY_OR_FAIL(expr)                                                                          \
    do {                                                                                           \
        cudaError_t e__ = (expr);                                                                  \
        if (e__ != cudaSuccess) {                                                                  \
            set_error("%s failed: %s", #expr, cudaGetErrorString(e__));                            \
            return fail(e__ == cudaErrorMemoryAllocation ? R3_ERR_ALLOC : R3_ERR_CUDA);            \
        }                                                                                          \
    } while (0)
    TRY_OR_FAIL(dev_malloc(&nb.X, sizeof(float) * B * (size_t)n1 * d));
    TRY_OR_FAIL(dev_malloc(&nb.y, sizeof(float) * B * (size_t)n1));
    TRY_OR_FAIL(dev_malloc(&nb.L64, sizeof(double) * B * mat1));
    TRY_OR_FAIL(dev_malloc(&nb.W64, sizeof(double) * B * mat1));
    TRY_OR_FAIL(dev_malloc(&nb.W32, sizeof(float) * B * mat1));
    TRY_OR_FAIL(dev_malloc(&nb.alpha64, sizeof(double) * B * np1));
    TRY_OR_FAIL(dev_malloc(&nb.alpha32, sizeof(float) * B * np1));
    TRY_OR_FAIL(dev_malloc(&nb.u, sizeof(double) * B * np1));
    TRY_OR_FAIL(dev_malloc(&nb.slabs, sizeof(double) * ((size_t)B + (size_t)B * kRowSlabs * np1)));
    TRY_OR_FAIL(dev_malloc(&nb.best, sizeof(float) * 2 * B));
    TRY_OR_FAIL(dev_malloc(&nb.wnorm, sizeof(double) * B));
    TRY_OR_FAIL(dev_malloc(&nb.scratch, factor_scratch_bytes(B, np1)));

    // histories: old rows then new rows, per GP
    TRY_OR_FAIL(cudaMemcpy2DAsync(nb.X, sizeof(float) * (size_t)n1 * d, gp->X, sizeof(float) * (size_t)n0 * d,
                                  sizeof(float) * (size_t)n0 * d, B, cudaMemcpyDeviceToDevice, stream));
    TRY_OR_FAIL(cudaMemcpy2DAsync(nb.X + (size_t)n0 * d, sizeof(float) * (size_t)n1 * d, Xnew,
                                  sizeof(float) * xnew_gp_stride, sizeof(float) * (size_t)k * d, B,
                                  cudaMemcpyDeviceToDevice, stream));
    TRY_OR_FAIL(cudaMemcpy2DAsync(nb.y, sizeof(float) * n1, gp->y, sizeof(float) * n0, sizeof(float) * n0, B,
                                  cudaMemcpyDeviceToDevice, stream));
    TRY_OR_FAIL(cudaMemcpy2DAsync(nb.y + n0, sizeof(float) * n1, ynew, sizeof(float) * ynew_gp_stride, sizeof(float) * k,
                                  B, cudaMemcpyDeviceToDevice, stream));
    const int kept = n0 / kFactorTile * kFactorTile;   // rows of whole tiles of old observations
    if (kept > 0) {
        embed_kernel<<<dim3(kept, B, 2), 128, 0, stream>>>(gp->L64, gp->W64, np0, nb.L64, nb.W64, np1, kept);
        ++g_launches;
        TRY_OR_FAIL(cudaGetLastError());
    }
    FactorProblem f;
    f.X = nb.X; f.y = nb.y; f.ell = gp->ell_d; f.sf2 = gp->sf2_d; f.sn2 = gp->sn2_d;
    f.batch = B; f.n = n1; f.d = d; f.npad = np1; f.rows_done = kept;
    f.L = nb.L64; f.W = nb.W64;
    f.best = nb.best; f.yabs = nb.best + B;
    r3_status_t st = factor_device(f, nb.scratch, gp->status_d, gp->device, stream);
    if (st != R3_OK) return fail(st);
    st = finish_weights(B, n1, np1, nb.W64, nb.y, nb.alpha64, nb.alpha32, nb.W32, nb.wnorm, nb.u, nb.slabs, stream);
    if (st != R3_OK) return fail(st);
    TRY_OR_FAIL(cudaMemcpyAsync(gp->status_h, gp->status_d, 2 * sizeof(int), cudaMemcpyDeviceToHost, stream));
    TRY_OR_FAIL(cudaStreamSynchronize(stream));
#undef TRY_OR_FAIL
    if (gp->status_h[0] & (DEV_NOT_PD | DEV_NONFINITE | DEV_TIMEOUT)) return fail(R3_OK);   // the caller reports; nothing swapped
    // success: the new arrays replace the old ones
    if (cudaMemcpy(gp->best_d, nb.best, sizeof(float) * B, cudaMemcpyDeviceToDevice) != cudaSuccess ||
        cudaMemcpy(gp->yabs_d, nb.best + B, sizeof(float) * B, cudaMemcpyDeviceToDevice) != cudaSuccess ||
        cudaMemcpy(gp->wnorm_d, nb.wnorm, sizeof(double) * B, cudaMemcpyDeviceToDevice) != cudaSuccess) {
        set_error("r3_gp_append: copying the incumbent failed");
        return fail(R3_ERR_CUDA);
    }
    dev_free(gp->X); dev_free(gp->y); dev_free(gp->L64); dev_free(gp->W64); dev_free(gp->W32);
    dev_free(gp->alpha64); dev_free(gp->alpha32);
    gp->X = nb.X; gp->y = nb.y; gp->L64 = nb.L64; gp->W64 = nb.W64; gp->W32 = nb.W32;
    gp->alpha64 = nb.alpha64; gp->alpha32 = nb.alpha32;
    nb.X = nullptr; nb.y = nullptr; nb.L64 = nullptr; nb.W64 = nullptr; nb.W32 = nullptr;
    nb.alpha64 = nullptr; nb.alpha32 = nullptr;
    nb.release();
    gp->n = n1;
    gp->npad = np1;
    return R3_OK;
}

}  // namespace r3
