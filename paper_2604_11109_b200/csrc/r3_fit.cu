// r3_gp_fit and r3_gp_append on the device: one upload, the factorisation (r3_factor.cu), the weights (r3_weights.cu), the
// tensor operands (r3_score_tc.cu), one read-back.
//
// Everything here runs once per BO round, in FP64, and is rounded to FP32 once at the end.  n is padded to a multiple of
// 32 with an identity block, which leaves L, W and alpha unchanged.
#include <limits.h>
#include <string.h>

#include <algorithm>

#include "r3_internal.cuh"

namespace r3 {

namespace {

// The block of small arrays: what the device reports first, then what it is told.
size_t carve_block(r3_fit_state& s, char* base, size_t* results)
{
    char* p = base;
    const size_t B = s.batch;
    auto take = [&](size_t bytes) {
        char* r = p;
        p += (bytes + 15) & ~(size_t)15;
        return r;
    };
    s.block = base;
    s.fit_status = (int*)take(4 * sizeof(int));
    s.best_d = (float*)take(sizeof(float) * B);
    s.yabs_d = (float*)take(sizeof(float) * B);
    s.wmax_d = (unsigned*)take(sizeof(unsigned) * B);
    s.xamax_d = (unsigned*)take(sizeof(unsigned));
    s.xnmax_d = (unsigned*)take(sizeof(unsigned) * B);
    s.wnorm_d = (double*)take(sizeof(double) * B);
    if (results) *results = (size_t)(p - base);
    s.ell_d = (float*)take(sizeof(float) * B * s.d);
    s.inv_ell = (float*)take(sizeof(float) * B * s.d);
    s.sf2_d = (float*)take(sizeof(float) * B);
    s.sn2_d = (float*)take(sizeof(float) * B);
    return (size_t)(p - base);
}

// Where an array of the device block lies in its host image
template <typename T>
T* mirror(const r3_fit_state& s, T* device, char* image) { return (T*)(image + ((char*)device - s.block)); }

#define TRY_ST(expr)                                                                               \
    do {                                                                                           \
        cudaError_t e__ = (expr);                                                                  \
        if (e__ != cudaSuccess) {                                                                  \
            set_error("%s failed: %s", #expr, cudaGetErrorString(e__));                            \
            return e__ == cudaErrorMemoryAllocation ? R3_ERR_ALLOC : R3_ERR_CUDA;                  \
        }                                                                                          \
    } while (0)

}  // namespace

r3_status_t state_alloc(r3_fit_state& s)
{
    s.npad = round_up(s.n, kFitBlock);
    const size_t B = s.batch, mat = (size_t)s.npad * s.npad;
    r3_fit_state layout = s;
    const size_t bytes = carve_block(layout, nullptr, nullptr);
    char* block = nullptr;
    TRY_ST(dev_malloc(&s.X, sizeof(float) * B * (size_t)s.n * s.d));
    TRY_ST(dev_malloc(&s.y, sizeof(float) * B * (size_t)s.n));
    TRY_ST(dev_malloc(&block, bytes));
    carve_block(s, block, nullptr);
    TRY_ST(dev_malloc(&s.L64, sizeof(double) * B * mat));
    TRY_ST(dev_malloc(&s.W64, sizeof(double) * B * mat));
    TRY_ST(dev_malloc(&s.W32, sizeof(float) * B * mat));
    TRY_ST(dev_malloc(&s.alpha64, sizeof(double) * B * s.npad));
    TRY_ST(dev_malloc(&s.alpha32, sizeof(float) * B * s.npad));
    return R3_OK;
}

void state_free(r3_fit_state& s)
{
    tc_release(s);
    dev_free(s.X);
    dev_free(s.y);
    dev_free(s.block);
    dev_free(s.L64);
    dev_free(s.W64);
    dev_free(s.W32);
    dev_free(s.alpha64);
    dev_free(s.alpha32);
    s = r3_fit_state();
}

r3_status_t state_fit(r3_gp* gp, r3_fit_state& s, int rows_done, bool full, bool need_tc, cudaStream_t stream, int* bits,
                      int* pivot, double* lml)
{
    const int B = s.batch, npad = s.npad;
    void* ints = nullptr;
    double* doubles = nullptr;
    auto done = [&](r3_status_t st) {
        // on an error something may still be in flight on the stream
        if (st != R3_OK) cudaStreamSynchronize(stream);
        FreeScope no_wait;
        dev_free(ints);
        dev_free(doubles);
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
    const size_t fbytes = factor_scratch_bytes(B, npad);
    TRY_DONE(dev_malloc(&ints, fbytes + sizeof(unsigned) * B));
    const size_t wdoubles = weights_scratch_doubles(B, npad);
    TRY_DONE(dev_malloc(&doubles, sizeof(double) * (wdoubles + (lml ? lml_scratch_doubles(s) : 0))));

    const bool own = &s == static_cast<r3_fit_state*>(gp);
    if (own) gp->fitted = false;
    // the block: results cleared, hyper-parameters filled in
    size_t results = 0;
    const size_t bytes = carve_block(s, s.block, &results);
    char* image = gp->stage_h;
    if (bytes > kStageBytes) {
        gp->image.resize(bytes);
        image = gp->image.data();
    }
    memset(image, 0, results);
    mirror(s, s.fit_status, image)[1] = INT_MAX;
    memcpy(mirror(s, s.ell_d, image), gp->ell.data(), sizeof(float) * gp->ell.size());
    float* inv = mirror(s, s.inv_ell, image);
    for (size_t i = 0; i < gp->ell.size(); ++i) inv[i] = (float)(1.0 / (double)gp->ell[i]);
    memcpy(mirror(s, s.sf2_d, image), gp->sf2.data(), sizeof(float) * B);
    memcpy(mirror(s, s.sn2_d, image), gp->sn2.data(), sizeof(float) * B);
    TRY_DONE(cudaMemcpyAsync(s.block, image, bytes, cudaMemcpyHostToDevice, stream));

    FactorProblem f;
    f.X = s.X; f.y = s.y; f.ell = s.ell_d; f.sf2 = s.sf2_d; f.sn2 = s.sn2_d;
    f.batch = B; f.n = s.n; f.d = s.d; f.npad = npad; f.rows_done = rows_done;
    f.L = s.L64; f.W = s.W64;
    f.best = s.best_d; f.yabs = s.yabs_d;
    f.wait = wait_rule(gp, STALL_FACTOR);
    r3_status_t st = factor_device(f, ints, B, s.fit_status, gp->device, stream);
    if (st != R3_OK) return done(st);
    WeightProblem w;
    w.W = s.W64; w.y = s.y;
    w.batch = B; w.n = s.n; w.npad = npad;
    w.alpha64 = s.alpha64; w.alpha32 = s.alpha32;
    w.W32 = full ? s.W32 : nullptr;
    w.wnorm = full ? s.wnorm_d : nullptr;
    w.wmax = full ? s.wmax_d : nullptr;
    w.wait = wait_rule(gp, STALL_WEIGHTS);
    st = weights_device(w, doubles, (unsigned*)((char*)ints + fbytes), s.fit_status, gp->device, stream);
    if (st != R3_OK) return done(st);
    if (full) {
        if (s.tc) {   // a refit: calls that still use the old operands end first
            cudaDeviceSynchronize();
            FreeScope no_wait;
            tc_release(s);
        }
        if (tc_supported(s.n, s.d)) {
            st = tc_prepare(s, gp->device, stream);
            s.tc_short = st == R3_ERR_ALLOC;
            if (st != R3_OK && (need_tc || st != R3_ERR_ALLOC)) return done(st);
        }
    }
    // the evidence goes behind the block's image if there is room
    const size_t lml_bytes = sizeof(double) * (size_t)B * (s.d + 3);
    const bool staged = lml && image == gp->stage_h && bytes + lml_bytes <= kStageBytes;
    if (lml) {
        double* out = nullptr;
        st = lml_enqueue(s, doubles + wdoubles, &out, s.fit_status, stream);
        if (st != R3_OK) return done(st);
        TRY_DONE(cudaMemcpyAsync(staged ? (void*)(image + bytes) : (void*)lml, out, lml_bytes, cudaMemcpyDeviceToHost, stream));
    }
    TRY_DONE(cudaMemcpyAsync(image, s.block, results, cudaMemcpyDeviceToHost, stream));
    TRY_DONE(cudaStreamSynchronize(stream));
    if (staged) memcpy(lml, image + bytes, lml_bytes);
#undef TRY_DONE
    const int* fs = mirror(s, s.fit_status, image);
    *bits = fs[0];
    if (pivot) *pivot = fs[1];
    if (fs[0] & DEV_BOUNDS) {
        set_error("bounds-checking build: an index check of the fit failed (source line %d of its kernel's file)", fs[2]);
        return done(R3_ERR_CUDA);
    }
    if (fs[0] & DEV_TIMEOUT) {
        set_error("a bounded device-side wait of the fit ran out");
        return done(R3_ERR_DEVICE_TIMEOUT);
    }
    if (full) {
        s.best.assign(mirror(s, s.best_d, image), mirror(s, s.best_d, image) + B);
        s.y_absmax.assign(mirror(s, s.yabs_d, image), mirror(s, s.yabs_d, image) + B);
        s.wnorm.assign(mirror(s, s.wnorm_d, image), mirror(s, s.wnorm_d, image) + B);
        if (s.tc && !tc_accept(s, gp->sf2.data(), mirror(s, s.wmax_d, image), *mirror(s, s.xamax_d, image))) {
            FreeScope no_wait;   // nothing has used them yet
            tc_release(s);
        }
        if (own) gp->fitted = !(fs[0] & (DEV_NOT_PD | DEV_NONFINITE));
    }
    return done(R3_OK);
}

// =====================================================================================================
// r3_gp_append: k more observations per GP without refactoring what is already factored.  The rows of L and W of whole
// tiles of old observations are copied, the rows below are computed as a fit computes them (r3_factor.cu): O(k n^2)
// against the fit's O(n^3 / 3), and the result is the one a fit of the concatenated history gives.
namespace {

// The old state's part of the new one, per GP: rows [0, rows) of L and W into matrices with another leading dimension
// (blockIdx.z = 0, 1; the columns right of the copied triangle are zeroed by the factorisation, or lie within the copied
// width and are zero there), old and new rows of X and y (blockIdx.z = 2).
__global__ void embed_kernel(const double* __restrict__ L0, const double* __restrict__ W0, int np0, double* __restrict__ L1,
                             double* __restrict__ W1, int np1, int rows, const float* __restrict__ X0,
                             const float* __restrict__ Xnew, const float* __restrict__ y0, const float* __restrict__ ynew,
                             int n0, int k, int d, float* __restrict__ X1, float* __restrict__ y1)
{
    const int g = blockIdx.y;
    if (blockIdx.z == 2) {
        const size_t n1 = n0 + k, old = (size_t)n0 * d, all = n1 * d, step = (size_t)gridDim.x * blockDim.x;
        const size_t at = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
        for (size_t e = at; e < all; e += step)
            X1[g * all + e] = e < old ? X0[g * old + e] : Xnew[(size_t)g * k * d + (e - old)];
        for (size_t e = at; e < n1; e += step) y1[g * n1 + e] = e < (size_t)n0 ? y0[(size_t)g * n0 + e] : ynew[(size_t)g * k + (e - n0)];
        return;
    }
    const int i = blockIdx.x;
    if (i >= rows) return;
    const double* src = (blockIdx.z ? W0 : L0) + (size_t)g * np0 * np0 + (size_t)i * np0;
    double* dst = (blockIdx.z ? W1 : L1) + (size_t)g * np1 * np1 + (size_t)i * np1;
    for (int c = 2 * threadIdx.x; c < rows; c += 2 * blockDim.x)
        *reinterpret_cast<double2*>(dst + c) = *reinterpret_cast<const double2*>(src + c);
}

}  // namespace

// The new state's tensor operands did not fit beside the old state's: now that those are gone, once more.  If there is still no
// memory for them the append stands and the CUDA-core engine serves the handle (r3_gp_engine tells).
static r3_status_t operands_again(r3_gp* gp, cudaStream_t stream)
{
    r3_status_t st = tc_prepare(*gp, gp->device, stream);
    if (st != R3_OK) return st == R3_ERR_ALLOC ? R3_OK : st;
    gp->tc_short = false;
    if (!gp->tc) return R3_OK;
    std::vector<unsigned> wmax(gp->batch);
    unsigned xamax = 0;
    R3_CUDA_TRY(cudaMemcpyAsync(wmax.data(), gp->wmax_d, sizeof(unsigned) * gp->batch, cudaMemcpyDeviceToHost, stream));
    R3_CUDA_TRY(cudaMemcpyAsync(&xamax, gp->xamax_d, sizeof(unsigned), cudaMemcpyDeviceToHost, stream));
    R3_CUDA_TRY(cudaStreamSynchronize(stream));
    if (!tc_accept(*gp, gp->sf2.data(), wmax.data(), xamax)) {
        FreeScope no_wait;   // nothing has used them yet
        tc_release(*gp);
    }
    return R3_OK;
}

r3_status_t append_device(r3_gp* gp, const float* Xnew, const float* ynew, int k, cudaStream_t stream, int* bits, int* pivot)
{
    r3_fit_state s;
    s.batch = gp->batch;
    s.d = gp->d;
    s.n = gp->n + k;
    auto drop = [&](r3_status_t st) {
        cudaStreamSynchronize(stream);
        FreeScope no_wait;
        state_free(s);
        return st;
    };
    r3_status_t st = state_alloc(s);
    if (st != R3_OK) return drop(st);
    const int kept = gp->n / kFactorTile * kFactorTile;   // rows of whole tiles of old observations
    embed_kernel<<<dim3(std::max(kept, 64), s.batch, 3), 128, 0, stream>>>(gp->L64, gp->W64, gp->npad, s.L64, s.W64, s.npad,
                                                                           kept, gp->X, Xnew, gp->y, ynew, gp->n, k, s.d, s.X, s.y);
    ++g_launches;
    if (cudaError_t e = cudaGetLastError(); e != cudaSuccess) {
        set_error("launch of embed_kernel failed: %s", cudaGetErrorString(e));
        return drop(R3_ERR_CUDA);
    }
    st = state_fit(gp, s, kept, true, false, stream, bits, pivot);
    if (st != R3_OK || (*bits & (DEV_NOT_PD | DEV_NONFINITE))) return drop(st);   // the caller reports; nothing swapped
    // success: the new state takes the old one's place (calls that still use the old one end first)
    cudaDeviceSynchronize();
    FreeScope no_wait;
    std::swap(static_cast<r3_fit_state&>(*gp), s);
    state_free(s);
    return gp->tc_short ? operands_again(gp, stream) : R3_OK;
}

}  // namespace r3
