// Internal declarations shared by the translation units of libr3gp (CUDA, sm_100a).
// Nothing here is part of the public ABI; see include/r3.h for that.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "r3.h"

namespace r3 {

// ---------------------------------------------------------------------------------------------
// error text (thread-local) and launch accounting
void set_error(const char* fmt, ...);
extern thread_local unsigned long long g_launches;

#define R3_CUDA_TRY(expr)                                                                \
    do {                                                                                 \
        cudaError_t e__ = (expr);                                                        \
        if (e__ != cudaSuccess) {                                                        \
            r3::set_error("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e__),       \
                          __FILE__, __LINE__);                                           \
            return e__ == cudaErrorMemoryAllocation ? R3_ERR_ALLOC : R3_ERR_CUDA;        \
        }                                                                                \
    } while (0)

// Launch a kernel, count it, and turn a launch error into a status.
#define R3_LAUNCH(kernel, grid, block, smem, stream, ...)                                \
    do {                                                                                 \
        kernel<<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__);                      \
        ++r3::g_launches;                                                                \
        cudaError_t e__ = cudaGetLastError();                                            \
        if (e__ != cudaSuccess) {                                                        \
            r3::set_error("launch of %s failed: %s (%s:%d)", #kernel,                    \
                          cudaGetErrorString(e__), __FILE__, __LINE__);                  \
            return R3_ERR_CUDA;                                                          \
        }                                                                                \
    } while (0)

// Bits of the device status word (one int per handle, OR-ed by kernels).
enum : int {
    DEV_NONFINITE = 1,   // NaN/Inf met in an input
    DEV_NOT_PD = 2,      // non-positive Cholesky pivot
    DEV_TIMEOUT = 4,     // a bounded wait gave up
    DEV_BOUNDS = 8,      // an index check of the bounds-checking build failed (R3_BOUNDS_CHECK)
};

// Index checks of the bounds-checking build (python -m paper_2604_11109_b200.build --check; compute-sanitizer is
// not available where this library is developed).  R3_IDX(i, n, status) is i in the normal build.  In the
// checking build an index outside [0, n) raises DEV_BOUNDS in the handle's status word, leaves the source line
// of the check in the word after the pivot index, and is replaced by 0: the access goes to a valid element
// instead of faulting, control flow stays as it was (warp-wide instructions keep all their lanes), and
// r3_gp_check reports the line.
#ifdef R3_BOUNDS_CHECK
__device__ __forceinline__ long long checked_index(long long i, long long n, int* status, int line)
{
    if (i >= 0 && i < n) return i;
    atomicOr(status, DEV_BOUNDS);
    atomicMax(status + 2, line);
    return 0;
}
#define R3_IDX(i, n, status) r3::checked_index((long long)(i), (long long)(n), (status), __LINE__)
#else
#define R3_IDX(i, n, status) (i)
#endif

constexpr int kFitBlock = 32;   // Cholesky / inverse block size; n is padded to a multiple of it
constexpr int kMaxN = 8192;
constexpr int kMaxD = 256;
constexpr int kMaxK = 1024;
constexpr int kAppendMax = 128;   // observations per r3_gp_append call

// device-memory cache (r3_alloc.cu): cudaMalloc/cudaFree with freed blocks kept for reuse
cudaError_t dev_malloc_bytes(void** p, size_t bytes);
template <typename T>
inline cudaError_t dev_malloc(T** p, size_t bytes)
{
    return dev_malloc_bytes(reinterpret_cast<void**>(p), bytes);
}
void dev_free(void* p);
// While one lives, dev_free on this thread does not wait for the device: whoever opens it knows that nothing in flight
// still uses what is freed (temporaries after their stream has been synchronised).
struct FreeScope {
    FreeScope();
    ~FreeScope();
    FreeScope(const FreeScope&) = delete;
    FreeScope& operator=(const FreeScope&) = delete;
};
void trim_cache();
constexpr int kPinnedInts = 1024;
constexpr int kStageInt = 128;       // where a handle's staging area begins in its pinned block
constexpr size_t kStageBytes = sizeof(int) * (kPinnedInts - kStageInt);
int* pinned_word_acquire();          // kPinnedInts pinned host ints from a process-wide pool (nullptr on failure)
void pinned_word_release(int* w);
size_t cached_bytes();

// Waits of a kernel whose blocks wait for one another: they give up after `cycles` (about two seconds unless a test asks for
// less); withhold (r3_gp_test_stall): one block keeps back what the others wait for.
constexpr long long kGridWaitCycles = 4000000000ll;
struct WaitRule {
    long long cycles = kGridWaitCycles;
    int withhold = 0;
};

inline int round_up(int a, int b) { return (a + b - 1) / b * b; }
inline long long round_up_ll(long long a, long long b) { return (a + b - 1) / b * b; }

}  // namespace r3

// A top-k that rides on the next scoring call of a handle: the guard kernel, which runs over the final EI
// anyway, leaves the k largest of each of its slices, and the selection's later levels follow at once.
struct TopkRequest {
    int k = 0;                 // 0: none
    int* idx = nullptr;        // device [batch][k]
    float* val = nullptr;      // device [batch][k] or nullptr
    void* ws = nullptr;        // at least guard_topk_workspace_bytes(batch, m, k)
    size_t ws_bytes = 0;
};

// Everything a fit produces.  A handle is one of these and what goes with it; r3_gp_append builds the next one beside
// the handle's and puts it in its place.
struct r3_fit_state {
    int batch = 0, n = 0, d = 0;
    int npad = 0;              // n rounded up to kFitBlock; padded rows/cols are identity / zero
    std::vector<float> best, y_absmax;        // host copies [batch]: incumbent, max |y|
    std::vector<double> wnorm;                // [batch] estimate of |L^-1|_2 (power iteration x 1.5)

    float* X = nullptr;        // [batch][n][d]   raw observations (FP32 as given)
    float* y = nullptr;        // [batch][n]      observed values as given (kept for r3_gp_append)
    double* L64 = nullptr;     // [batch][npad][npad] lower Cholesky factor (upper part zero)
    double* W64 = nullptr;     // [batch][npad][npad] W = L^-1, lower
    float* W32 = nullptr;      // [batch][npad][npad] W rounded to FP32
    double* alpha64 = nullptr; // [batch][npad]  (zero in the padding)
    float* alpha32 = nullptr;  // [batch][npad]

    // the small arrays, in one block that a fit uploads and whose first part it reads back
    char* block = nullptr;
    int* fit_status = nullptr; // [4] status bits, first bad pivot index
    float* best_d = nullptr;   // [batch]
    float* yabs_d = nullptr;   // [batch] max |y|
    unsigned* wmax_d = nullptr;   // [batch] bits of max |W|
    unsigned* xamax_d = nullptr;  // bits of the largest scaled coordinate
    unsigned* xnmax_d = nullptr;  // [batch] bits of max |x~|^2
    double* wnorm_d = nullptr; // [batch]
    float* ell_d = nullptr;    // [batch][d]      lengthscales as given
    float* inv_ell = nullptr;  // [batch][d]      1/lengthscale
    float* sf2_d = nullptr;    // [batch]
    float* sn2_d = nullptr;    // [batch]

    // tensor-core operands (built by the fit when the tensor engine can serve (n, d))
    void* tc = nullptr;        // r3::TensorOperands*, see r3_score_tc.cu
    bool tc_short = false;     // they are missing because there was no memory for them
};

// The handle.  Device arrays are allocated at fit time and freed by r3_gp_free.
struct r3_gp : r3_fit_state {
    int device = 0;
    bool fitted = false;       // factor, weights and operands belong together; false while a refit is under way or has failed
    std::vector<float> ell, sf2, sn2;         // host copies [batch][d], [batch], [batch]
    int* status_d = nullptr;   // [4]: status bits of the scoring calls, pivot, line of a failed index check, unused
    int* status_h = nullptr;   // pinned mirror of status_d
    int* rescued_h = nullptr;  // pinned [64]: candidates recomputed in FP64 by the last scoring call, per GP
    char* stage_h = nullptr;   // pinned [kStageBytes]: uploads and read-backs of a fit's block
    std::vector<char> image;   // the same for blocks that do not fit there

    // grow-only private workspace used by scoring and top-k
    void* ws = nullptr;
    size_t ws_bytes = 0;

    r3_engine_t engine_req = R3_ENGINE_AUTO;
    TopkRequest topk_req;      // set by r3_gp_score_topk for the scoring call it makes, consumed by the guard

    // bounded device-side waits of the tensor engine: the limit in cycles, and the test aid that makes one run out
    long long wait_limit_cycles = 4000000000ll;   // about 2 s
    long long withhold_w = -1;
    int stall_where = -1;             // r3_gp_test_stall: the kernel, and the limit of its waits
    long long stall_cycles = 0;

    // optional timing of the dominant scoring kernel: event pairs recorded around its launches
    bool profile = false;
    std::vector<cudaEvent_t> events;   // pairs (start, stop)
    size_t events_used = 0;

    // the host-buffer entry point copies the pool in pieces on a stream of its own while earlier pieces are scored
    cudaStream_t copy_stream = nullptr;
    std::vector<cudaEvent_t> copy_events;
};

namespace r3 {

// The rule for the next launch of kernel `where`; a test's request holds for one launch.
enum : int { STALL_FACTOR = 0, STALL_WEIGHTS = 1, STALL_GUARD = 2, STALL_PROPOSE = 3 };
WaitRule wait_rule(r3_gp* gp, int where);

// factor and inverse factor (r3_factor.cu)
constexpr int kFactorTile = 64;
struct FactorProblem {
    const float *X, *y, *ell, *sf2, *sn2;   // [batch][n][d], [batch][n], [batch][d], [batch], [batch]
    int batch, n, d, npad;
    int rows_done;          // rows of L and W that are there already: a multiple of kFactorTile
    double *L, *W;          // [batch][npad][npad]
    float *best, *yabs;     // [batch] min y, max |y|
    WaitRule wait;
};
size_t factor_scratch_bytes(int batch, int npad);
// Asynchronous; non-finite inputs and non-positive pivots are latched in `status`.
// `scratch`: factor_scratch_bytes, followed by extra_ints more ints that are cleared with it.
r3_status_t factor_device(const FactorProblem& p, void* scratch, int extra_ints, int* status, int device, cudaStream_t stream);

// weights, norm estimate and FP32 copy of the inverse factor (r3_weights.cu)
struct WeightProblem {
    const double* W;        // [batch][npad][npad]
    const float* y;         // [batch][n]
    int batch, n, npad;
    double* alpha64;        // [batch][npad]
    float* alpha32;         // [batch][npad]
    float* W32;             // [batch][npad][npad], or nullptr
    double* wnorm;          // [batch], or nullptr: weights only
    unsigned* wmax;         // [batch] bits of max |W|, zero on entry, or nullptr
    WaitRule wait;
};
size_t weights_scratch_doubles(int batch, int npad);
// barrier: [batch] words, zero on entry.  Asynchronous.
r3_status_t weights_device(const WeightProblem& p, double* scratch, unsigned* barrier, int* status, int device,
                           cudaStream_t stream);

// fit (r3_fit.cu)
r3_status_t state_alloc(r3_fit_state& s);    // arrays for s.batch, s.n, s.d
void state_free(r3_fit_state& s);
// The fit of s (histories in place, hyper-parameters from gp's host copies), rows below rows_done of L and W given.
// full: everything a handle needs, tensor operands included; otherwise L, W, alpha and the status only (an evaluation of
// the evidence, which leaves the handle without a fit).  Synchronises; *bits and *pivot are what the device found.  need_tc: a failed allocation of the tensor
// operands is an error (otherwise the CUDA-core engine serves the state).
// lml: if not nullptr receives the evidence and its gradient, host [batch][d + 3] (meaningless when *bits reports a failure).
r3_status_t state_fit(r3_gp* gp, r3_fit_state& s, int rows_done, bool full, bool need_tc, cudaStream_t stream, int* bits,
                      int* pivot, double* lml = nullptr);
// Appends k observations per GP (r3_gp_append): extends L, W, alpha, X, y in O(k n^2); synchronises.  On
// any error (and when *bits says so) the handle is left as it was.
r3_status_t append_device(r3_gp* gp, const float* Xnew, const float* ynew, int k, cudaStream_t stream, int* bits, int* pivot);

// SIMT scoring (r3_score_simt.cu)
size_t score_simt_workspace_bytes(const r3_gp* gp, long long m);
r3_status_t score_simt(r3_gp* gp, const float* Xcand, long long m, float* mu, float* sigma, float* ei,
                       void* ws, size_t ws_bytes, cudaStream_t stream);

// Accuracy guard and FP64 rescue (r3_rescue.cu).  The engines write their results and, per candidate,
// estimates of their own rounding error in mu (err_mu) and in q = |W k*|^2 (err_q); the guard then
// lists the candidates that may miss the accuracy contract and recomputes them in FP64.
struct GuardBuffers {
    float* err_mu;      // [batch][m]
    float* err_q;       // [batch][m]
    int* list;          // [batch][m] candidates to recompute
    int* count;         // [batch] entries of the list
    int* total;         // [batch] candidates flagged
    unsigned* maxbits;  // [batch] bit pattern of the largest EI
    unsigned* done;     // [batch] slices selected
    unsigned* barrier;  // grid barrier of the guard kernel
    int* mode;          // what guard_pilot decided
    double *ks, *qpart, *mupart;   // the rescue's slab
};
size_t guard_workspace_bytes(const r3_gp* gp, long long m);
// The pool's maximum EI and the guard kernel's counters start at zero: the engines' first kernel of a pool clears this
// many ints from GuardBuffers::count on.
int guard_zero_ints(const r3_gp* gp);
// Key storage the guard kernel needs to leave the first level of a top-k of k (see TopkRequest).
size_t guard_topk_workspace_bytes(int batch, long long m, int k);
// Looks at the first `rows` scored candidates and decides (b.mode, on the device) whether so many of them miss the accuracy
// contract that the engine should score the pool in its more accurate form.
r3_status_t guard_pilot(r3_gp* gp, long long m, long long rows, const GuardBuffers& b, const float* mu, const float* sigma,
                        const float* ei, cudaStream_t stream);
GuardBuffers guard_carve(const r3_gp* gp, long long m, void* ws);
// have_max: the engine has raised maxbits to the pool's largest EI; tile_max: it has left the largest of each tile instead, one per 32 rows
r3_status_t guard_and_rescue(r3_gp* gp, const float* Xcand, long long m, const GuardBuffers& b, float* mu,
                             float* sigma, float* ei, const float* tile_max, long long tiles_per_gp, bool have_max, cudaStream_t stream);

// tensor-core scoring (r3_score_tc.cu)
bool tc_supported(int n, int d);
// Allocates the tensor operands of a state whose weights are under way on `stream` and launches their preparation;
// s.tc stays nullptr when no shape fits.  tc_accept, after the stream has been synchronised and the block read back:
// false when the values do not suit the FP16 planes (the caller releases the operands and the CUDA-core engine serves).
r3_status_t tc_prepare(r3_fit_state& s, int device, cudaStream_t stream);
bool tc_accept(const r3_fit_state& s, const float* sf2, const unsigned* wmax, unsigned xamax);
void tc_release(r3_fit_state& s);
void tc_info(const r3_gp* gp, int* info);   // r3_gp_tensor_info
size_t score_tc_workspace_bytes(const r3_gp* gp, long long m);
r3_status_t score_tc(r3_gp* gp, const float* Xcand, long long m, float* mu, float* sigma, float* ei,
                     void* ws, size_t ws_bytes, cudaStream_t stream);
// The same in pieces, for a caller that overlaps the pool's copy with the scoring: tiles [tile_begin, tile_end) of
// the score_tc_tiles(gp, m) tiles of 128 candidates (tile_end < 0: all of them), the guard optionally left to
// one score_tc_guard call after the last piece.
long long score_tc_tiles(const r3_gp* gp, long long m);
// tiles at the pool's beginning that are scored ahead of the others (0: none)
long long score_tc_first_tiles(const r3_gp* gp, long long m);
bool score_tc_can_split(const r3_gp* gp);
r3_status_t score_tc_part(r3_gp* gp, const float* Xcand, long long m, float* mu, float* sigma, float* ei, void* ws,
                          size_t ws_bytes, long long tile_begin, long long tile_end, bool guard, cudaStream_t stream);
r3_status_t score_tc_guard(r3_gp* gp, const float* Xcand, long long m, float* mu, float* sigma, float* ei, void* ws,
                           cudaStream_t stream);

// top-k (r3_topk.cu)
size_t topk_workspace_bytes(int batch, long long m, int k);
r3_status_t topk_finish_from_keys(unsigned long long* keys_in, unsigned long long* keys_tmp, int batch, long long count,
                                  int k, const float* ei, long long m, int* idx, float* val, cudaStream_t stream);
r3_status_t topk_device(const float* ei, int batch, long long m, int k, int* idx, float* val, void* ws,
                        size_t ws_bytes, cudaStream_t stream);

// log marginal likelihood and gradient (r3_lml.cu): out_h host [batch][d + 3]
size_t lml_scratch_doubles(const r3_fit_state& s);
r3_status_t lml_enqueue(const r3_fit_state& s, double* scratch, double** out, int* status, cudaStream_t stream);
r3_status_t lml_device(r3_gp* gp, double* out_h, cudaStream_t stream);

// greedy batch proposal on a shortlist (r3_propose.cu)
size_t propose_workspace_bytes(int batch, int npad, int R, int q);
r3_status_t propose_shortlist(r3_gp* gp, const float* Xcand, long long m, const int* sidx, const float* sval, int Rk, int R,
                              int q, int liar, int* idx_out, float* ei_out, int** cert, void* ws, cudaStream_t stream);

// fixed (never allocated) key storage for r3_topk_noalloc
r3_status_t topk_static_scratch(void** ptr);
size_t topk_static_capacity_keys();
size_t topk_static_capacity_bytes();

r3_status_t ensure_workspace(r3_gp* gp, size_t bytes);

// Event pair around one launch of the dominant kernel (no-ops unless profiling is on).
void prof_begin(r3_gp* gp, cudaStream_t stream);
void prof_end(r3_gp* gp, cudaStream_t stream);

}  // namespace r3
