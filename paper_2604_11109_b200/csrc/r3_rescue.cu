// What follows a pool's scoring, in one cooperatively launched kernel: the pool's largest EI, the accuracy guard,
// the FP64 rescue pass and the selection.
//
// The scoring engines work at FP32 level.  That is enough for almost every candidate of a
// well-conditioned GP, but not where the posterior variance sf2 - |W k*|^2 is a small difference of
// two numbers close to sf2 (a candidate on top of an observation), nor where mu = k*.alpha cancels
// heavily (an ill-conditioned history with large weights).  Each engine therefore writes, next to
// its results, an estimate of its own rounding error in mu and in q.  Once the whole pool is scored, guard_kernel
//   finds    the pool's largest EI (the EI tolerance is relative to it), unless the engine already has or has left the largest of
//            each of its tiles, of which every block takes the largest by itself (a pass over the pool and a grid barrier less),
//   flags    the candidates whose estimated error exceeds half of the accuracy contract
//            (1e-4 relative on mu and sigma with absolute floors, 1e-5 max(EI) on EI) in a list per GP,
//   rescues  them: recomputes them from the raw inputs entirely in FP64 -- direct-difference distances with
//            FP64 reciprocal lengthscales, FP64 weights and the FP64 inverse factor -- and overwrites
//            their mu, sigma and EI,
//   selects  (when the call asked for a top-k) the k largest final EI of every slice of the pool as 64-bit keys; when
//            a GP's slices leave at most 4096 keys the block that finishes its last slice writes the answer,
//            otherwise r3_topk.cu goes on from the keys.
//
// The rescue is a matrix product, V = W Ks with Ks the FP64 cross-covariance of all listed candidates, of which only
// the column sums of squares are kept.  Blocks compute Ks into a slab of the workspace, meet at a grid barrier, and
// share out (64 rows of W) x (64 candidates) tiles that run on the FP64 tensor path.  Few listed candidates (less
// than two tiles per block) get 16 x 16 tiles instead, whose reductions the block's eight warps split, so that W is
// read once by the whole GPU.  With at most 128 observations a block recomputes the first 16 it flags in a slice by
// itself, which saves a small call the barriers.  Whole calls, by the flagging block and by all blocks, on 4096 and on 65,536
// candidates of 16 features: 64 observations 37.1 | 43.6 and 70.2 | 76.4 us, 96 (none and 15 flagged) 30.9 | 31.1 and
// 72.3 | 74.9, 128 45.6 | 47.7 and 79.2 | 82.2, 160 51.4 | 49.7 and 98.9 | 96.9, 192 51.8 | 49.7 and 107.0 | 104.9,
// 256 59.5 | 51.7 and 127.5 | 117.4.  (A pool of which a third is flagged loses a little at 96: 65.0 | 60.8.)
// Bound: the FP64 rate for long lists, one read of W otherwise.  Measured, before (the block that met a flagged candidate
// recomputed it alone, four at a time) and now: 65,536 candidates at n = 4096, most of them listed, 300-600 ms and
// 36 ms (31 TFLOP/s of FP64); 2222 candidates at n = 701 1.50 ms and 0.14 ms; one pool of 262,144 with four listed
// (n = 256) 54 us and 33 us; 64 pools of 65,536 with three listed (n = 512) 318 us (with the kernel that found the
// largest EI) and 201 us.
#include <algorithm>

#include "r3_cross.cuh"
#include "r3_epilogue.cuh"
#include "r3_internal.cuh"
#include "r3_topk.cuh"

namespace r3 {

namespace {

constexpr int kThreads = kCrossThreads;
constexpr int kTile = kCrossTile;   // rows of W and candidates of a tile of the long-list form
constexpr int kSmallTile = 16;   // of the short-list form
constexpr size_t kSlabBytes = 64ull << 20;   // FP64 cross-covariances in flight: they stay in L2 beside W
constexpr int kOwnMaxN = 128;                // histories whose flagged candidates the flagging block recomputes itself
constexpr size_t kOwnKs = 12 * 1024;         // byte offset of its k* behind the staged coordinates (11.5 KB)
constexpr size_t kMaxSmem = 80 * 1024;       // operand stages (60 KB) and the tile prefix of 4096 GPs
constexpr int kFinishKeys = 4096;            // a GP whose slices leave at most this many keys is finished in the kernel

struct GuardArgs {
    const float *X, *ell, *sf2v, *bestv, *yabsv, *Xcand;
    const double *alpha64, *W64;
    int batch, n, d, npad;
    long long m;
    int chunk, chunks_per_gp;     // candidates a block looks over at a time (largest EI, flags)
    int slice, slices_per_gp;     // candidates of which a block selects the k largest, a multiple of a chunk; at most 4096
    float *mu, *sigma, *ei;
    const float *err_mu, *err_q;
    int* list;                    // [batch][m] flagged candidates of each GP
    unsigned* maxbits;            // [batch] bit pattern of the pool's largest EI
    int* count;                   // [batch] candidates in the list
    int* total;                   // [batch] candidates flagged (and recomputed)
    int* rescued_h;               // pinned host [64]: the same for the caller
    unsigned* done;               // [batch] slices selected so far
    unsigned* barrier;            // grid barrier
    int* status;                  // the handle's status words
    WaitRule wait;
    bool have_max;                // maxbits holds the largest EI already, or tile_max does:
    const float4* tile_max;       // [batch][tiles_per_gp] the engine's largest EI of each tile, one per 32 rows, or nullptr
    int tiles_per_gp;
    double *ks, *qpart, *mupart;  // slab: [slab][npad], [slab][npad / 16], [slab][ceil(npad / 64)]
    int slab;                     // candidates per slab, a multiple of 64
    int k, K2;                    // top-k request (k = 0: none); K2 = min(k, slice): keys a slice yields
    unsigned select_offset;       // byte offset of the selection's scratch in the dynamic shared memory
    unsigned pref_offset;         // byte offset of the tile prefix
    unsigned long long* keys;     // [batch][slices_per_gp][K2]
    bool finish;                  // the last slice of a GP writes the answer
    int* idx;
    float* val;
};

// Whether a candidate's estimated errors may exceed half of the accuracy contract.
__device__ __forceinline__ bool misses_contract(float mu, float sd, float dmu, float dq, float tol_ei, float mu_floor,
                                                float sd_floor, float best, float sf2)
{
    // d sigma = dq / (2 sigma); with sigma -> 0 every rounding error in q matters
    const float dsd = (sd > 0.f) ? dq / (2.f * sd) : ((dq > 0.f) ? INFINITY : 0.f);
    const float tol_mu = 1e-4f * fabsf(mu) + mu_floor;
    const float tol_sd = 1e-4f * sd + sd_floor;
    bool flag = !(dmu <= 0.5f * tol_mu) || !(dsd <= 0.5f * tol_sd);
    // EI: dEI = Phi(z) dmu + phi(z) dsigma against 1e-5 of the pool's largest EI.  Phi(z) <= exp(-z^2/2) / 2 for z <= 0 (and
    // <= 1 above) and phi(z) < 0.4 exp(-z^2/2): most candidates pass by that bound and need no erfc.
    const float z = (sd > 0.f) ? (best - mu) / sd : 0.f;
    const float bell = expf(-0.5f * z * z);
    if (isfinite(dsd) && !((z > 0.f ? dmu : 0.501f * bell * dmu) + 0.4f * bell * dsd <= 0.5f * tol_ei)) {
        const float Phi = 0.5f * erfcf(-z * 0.70710678f);
        flag |= !(Phi * dmu + bell * 0.39894228f * dsd <= 0.5f * tol_ei);
    }
    flag |= !(sd * sd >= 1e-3f * sf2);   // deep cancellation: do not trust the estimates either
    return flag;
}

// One block looks at the first `rows` candidates (GP after GP) of a pool that the engine has scored in its cheaper form:
// mode <- 1 when more than one in 32 of them would have to be recomputed, 0 otherwise.  The test is the guard's except that EI
// is measured against the largest in the sample, over all its GPs: of a GP on a smaller scale than another's it sees errors of
// mu and sigma only (which decide on the pools that were tried: two GPs a factor of 1e4 apart got the decision that equal
// scales get).  One decision serves the whole pool, whatever lies behind the sample.  Clears the guard's counters.
__global__ void __launch_bounds__(1024) pilot_kernel(const GuardArgs a, long long rows, int* __restrict__ mode, int* __restrict__ zero,
                                                     int zeros)
{
    __shared__ unsigned top_s;
    __shared__ int count_s;
    const int t = threadIdx.x;
    for (int i = t; i < zeros; i += 1024) zero[i] = 0;
    if (t == 0) {
        top_s = 0u;
        count_s = 0;
    }
    __syncthreads();
    float v = 0.f;
#pragma unroll 8
    for (long long f = t; f < rows; f += 1024) v = fmaxf(v, a.ei[f]);
    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
    if (t % 32 == 0) atomicMax(&top_s, top);
    __syncthreads();
    const float tol_ei = 1e-5f * __uint_as_float(top_s);
    int mine = 0;
#pragma unroll 4
    for (long long f = t; f < rows; f += 1024) {
        const int g = (int)(f / a.m);
        const float sf2 = a.sf2v[g];
        mine += misses_contract(a.mu[f], a.sigma[f], a.err_mu[f], a.err_q[f], tol_ei, 1e-6f * a.yabsv[g], 1e-6f * sqrtf(sf2),
                                a.bestv[g], sf2) ? 1 : 0;
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (t % 32 == 0 && mine) atomicAdd(&count_s, mine);
    __syncthreads();
    if (t == 0) *mode = (long long)count_s * 32 > rows ? 1 : 0;
}

__device__ __forceinline__ const float* cand_row(const GuardArgs& a, int g, int cand)
{
    return a.Xcand + (size_t)R3_IDX((long long)g * a.m + cand, (long long)a.batch * a.m, a.status) * a.d;
}

__device__ __forceinline__ void write_result(const GuardArgs& a, int g, int cand, double mu, double q)
{
    const size_t f = (size_t)R3_IDX((long long)g * a.m + cand, (long long)a.batch * a.m, a.status);
    const CandidateResult res = finalize_candidate(mu, q, (double)a.sf2v[g], (double)a.bestv[g]);
    a.mu[f] = res.mu;
    a.sigma[f] = res.sigma;
    a.ei[f] = res.ei;
}

// 64 rows of W times 64 candidates: column sums of squares to qpart[slot][rt].
__device__ __forceinline__ void rescue_tile(const GuardArgs& a, const double* __restrict__ Wg, size_t slot0, int rt,
                                            unsigned char* smem)
{
    const int t = threadIdx.x, w = t / 32, l = t % 32, wn = (w / 4) * 32;
    const int npad = a.npad, i0 = rt * kTile;
    double c[2][4][2] = {};
    // W is lower triangular: columns up to the tile's last row
    nt_tile(Wg + (size_t)i0 * npad, npad - i0, a.ks + (size_t)R3_IDX(slot0, a.slab - (kTile - 1), a.status) * npad, kTile, npad,
            min(npad, i0 + kTile), smem, c, a.status);
    double* red = reinterpret_cast<double*>(smem);        // [4 row warps][64 candidates]
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            double s = fma(c[0][j][h], c[0][j][h], c[1][j][h] * c[1][j][h]);
            for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (l < 4) red[(w % 4) * kTile + wn + j * 8 + 2 * l + h] = s;
        }
    __syncthreads();
    if (t < kTile)
        a.qpart[(slot0 + t) * (npad / 16) + rt] = (red[t] + red[kTile + t]) + (red[2 * kTile + t] + red[3 * kTile + t]);
}

// 16 rows of W times 16 candidates, the reduction split over the block's eight warps; operands straight from L2.
// Within a group of eight k the lanes hold pairs (2 l, 2 l + 1): the two products of a pair take the even and the odd
// k, for both operands alike.
__device__ __forceinline__ void rescue_small_tile(const GuardArgs& a, const double* __restrict__ Wg, size_t slot0, int rt,
                                                  unsigned char* smem)
{
    double* red = reinterpret_cast<double*>(smem);        // [8 warps][16][17], then [16][17]
    const int t = threadIdx.x, w = t / 32, l = t % 32;
    const int npad = a.npad, i0 = rt * kSmallTile;
    const int groups = min(npad, (i0 + kSmallTile + 7) / 8 * 8) / 8;
    const double* wa = Wg + (size_t)(i0 + l / 4) * npad + 2 * (l % 4);
    const double* kb = a.ks + ((size_t)R3_IDX(slot0, a.slab - (kSmallTile - 1), a.status) + l / 4) * npad + 2 * (l % 4);
    double c[2][2][2] = {};
#pragma unroll 4
    for (int gk = w; gk < groups; gk += 8) {
        double2 fa[2], fb[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            fa[i] = __ldcg(reinterpret_cast<const double2*>(wa + (size_t)i * 8 * npad + gk * 8));
            fb[i] = __ldcg(reinterpret_cast<const double2*>(kb + (size_t)i * 8 * npad + gk * 8));
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                dmma(c[i][j], fa[i].x, fb[j].x);
                dmma(c[i][j], fa[i].y, fb[j].y);
            }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) red[(w * 16 + i * 8 + l / 4) * 17 + j * 8 + 2 * (l % 4) + h] = c[i][j][h];
    __syncthreads();
    const int row = t / 16, col = t % 16;
    double v = 0.0;
#pragma unroll
    for (int ww = 0; ww < 8; ++ww) v += red[(ww * 16 + row) * 17 + col];
    __syncthreads();
    red[row * 17 + col] = v * v;
    __syncthreads();
    if (t < kSmallTile) {
        double s = 0.0;
#pragma unroll
        for (int r = 0; r < 16; ++r) s += red[r * 17 + t];
        a.qpart[(slot0 + t) * (npad / 16) + rt] = s;
    }
}

// Every listed candidate recomputed in FP64, tiles of CT candidates, a slab of tiles at a time.  Returns false when a
// grid barrier ran out.
template <int CT>
__device__ __forceinline__ bool rescue(const GuardArgs& a, const int* pref, int tiles, unsigned& target, unsigned char* smem)
{
    const int nb = (a.npad + 63) / 64, row_tiles = (a.npad + CT - 1) / CT;
    const int slab_tiles = a.slab / CT;
    auto gp_of = [&](int tile) {   // last g with pref[g] <= tile
        int lo = 0, hi = a.batch - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (pref[mid] <= tile) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    for (int t0 = 0; t0 < tiles; t0 += slab_tiles) {
        const int nt = min(slab_tiles, tiles - t0);
        for (int item = blockIdx.x; item < nt * nb; item += gridDim.x) {
            const int tile = item % nt, g = gp_of(t0 + tile), first = (t0 + tile - pref[g]) * CT;
            const int* list_g = a.list + (size_t)g * a.m + first;
            const int kb = item / nt;
            const size_t slot0 = R3_IDX((size_t)tile * CT, a.slab - (CT - 1), a.status);
            const int in_tile = min(CT, __ldcg(a.count + g) - first);
            cross_tile<CT>(
                a.n, a.d, a.npad, a.ell + (size_t)g * a.d, (double)a.sf2v[g], a.alpha64 + (size_t)g * a.npad,
                [&](int r) { return r < in_tile ? cand_row(a, g, __ldcg(list_g + r)) : nullptr; },
                [&](int k) { return a.X + ((size_t)g * a.n + R3_IDX(k, a.n, a.status)) * a.d; }, kb, smem,
                [&](int c, int k, double kv) { a.ks[R3_IDX((slot0 + c) * a.npad + k, (size_t)a.slab * a.npad, a.status)] = kv; },
                [&](int c, double part) { a.mupart[R3_IDX((slot0 + c) * nb + kb, (size_t)a.slab * nb, a.status)] = part; });
        }
        if (!grid_barrier(a.barrier, target, a.status, a.wait)) return false;
        for (int item = blockIdx.x; item < nt * row_tiles; item += gridDim.x) {   // the longest rows first
            const int tile = item % nt, rt = row_tiles - 1 - item / nt;
            const double* Wg = a.W64 + (size_t)gp_of(t0 + tile) * a.npad * a.npad;
            if (CT == kTile) rescue_tile(a, Wg, (size_t)tile * CT, rt, smem);
            else rescue_small_tile(a, Wg, (size_t)tile * CT, rt, smem);
        }
        if (!grid_barrier(a.barrier, target, a.status, a.wait)) return false;
        for (int s = blockIdx.x * kThreads + threadIdx.x; s < nt * CT; s += gridDim.x * kThreads) {
            const int tile = s / CT, g = gp_of(t0 + tile), pos = (t0 + tile - pref[g]) * CT + s % CT;
            if (pos >= __ldcg(a.count + g)) continue;
            double mu = 0.0, q = 0.0;
#pragma unroll 4
            for (int b = 0; b < nb; ++b) mu += __ldcg(a.mupart + (size_t)s * nb + b);
#pragma unroll 4
            for (int r = 0; r < row_tiles; ++r) q += __ldcg(a.qpart + (size_t)s * (a.npad / 16) + r);
            write_result(a, g, __ldcg(a.list + (size_t)g * a.m + pos), mu, q);
        }
        // the next slab overwrites the partial sums that other blocks may still be adding up
        if (t0 + slab_tiles < tiles && !grid_barrier(a.barrier, target, a.status, a.wait)) return false;
    }
    return true;
}

// Short histories: the block that flags a candidate recomputes it at once, up to 16 per slice, without meeting the other
// blocks: k* of the tile in shared memory, every warp 8 rows of W times the 16 candidates at a time.
__device__ __forceinline__ void rescue_own(const GuardArgs& a, int g, const int* own, int count, unsigned char* smem)
{
    double* ks = reinterpret_cast<double*>(smem + kOwnKs);   // [16][npad + 8]: fragment reads on different banks
    const int ld = a.npad + 8;
    double* mu_s = ks + kSmallTile * ld;                      // [16]
    double* q_s = mu_s + kSmallTile;                          // [8][16]
    const int t = threadIdx.x, w = t / 32, l = t % 32;
    if (t < kSmallTile) mu_s[t] = 0.0;
    for (int kb = 0; kb < (a.npad + 63) / 64; ++kb)
        cross_tile<kSmallTile>(
            a.n, a.d, a.npad, a.ell + (size_t)g * a.d, (double)a.sf2v[g], a.alpha64 + (size_t)g * a.npad,
            [&](int r) { return r < count ? cand_row(a, g, own[r]) : nullptr; },
            [&](int k) { return a.X + ((size_t)g * a.n + R3_IDX(k, a.n, a.status)) * a.d; }, kb, smem, [&](int c, int k, double kv) { ks[R3_IDX(c * ld + k, kSmallTile * ld, a.status)] = kv; },
            [&](int c, double part) { mu_s[c] += part; });
    __syncthreads();
    const double* Wg = a.W64 + (size_t)g * a.npad * a.npad;
    double q[2][2] = {};
    for (int i0 = w * 8; i0 < a.npad; i0 += 64) {
        const double* wa = Wg + (size_t)(i0 + l / 4) * a.npad + 2 * (l % 4);
        const double* kb = ks + (l / 4) * ld + 2 * (l % 4);
        double c[2][2][2] = {};   // [even and odd k][candidates]
#pragma unroll 4
        for (int k = 0; k < i0 + 8; k += 8) {
            const double2 fa = *reinterpret_cast<const double2*>(wa + k);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const double2 fb = *reinterpret_cast<const double2*>(kb + j * 8 * ld + k);
                dmma(c[0][j], fa.x, fb.x);
                dmma(c[1][j], fa.y, fb.y);
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const double v = c[0][j][h] + c[1][j][h];
                q[j][h] = fma(v, v, q[j][h]);
            }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            double s = q[j][h];
            for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (l < 4) q_s[w * kSmallTile + j * 8 + 2 * l + h] = s;
        }
    __syncthreads();
    if (t < count) {
        double s = 0.0;
        for (int ww = 0; ww < 8; ++ww) s += q_s[ww * kSmallTile + t];
        write_result(a, g, own[t], mu_s[t], s);
    }
}

// What guard_kernel does; false: a barrier ran out.
__device__ __forceinline__ bool guard_pool(const GuardArgs& a, unsigned char* smem)
{
    __shared__ int own[kSmallTile], own_count;
    __shared__ int warp_sum[8];
    __shared__ bool last_slice;
    const int t = threadIdx.x, lane = t % 32, warp = t / 32;
    const long long m = a.m;
    const int slices = a.slices_per_gp * a.batch, chunks = a.chunks_per_gp * a.batch;
    const bool own_rescue = a.npad <= kOwnMaxN;
    unsigned target = 0;

    // ---- the pool's largest EI
    if (!a.have_max) {
        for (int s = blockIdx.x; s < chunks; s += gridDim.x) {
            const int g = s / a.chunks_per_gp;
            const long long c0 = (long long)(s % a.chunks_per_gp) * a.chunk, c1 = min(m, c0 + a.chunk);
            float v = 0.f;
#pragma unroll 8
            for (long long i = c0 + t; i < c1; i += kThreads) v = fmaxf(v, __ldcg(a.ei + (size_t)g * m + i));  // EI >= 0; fmaxf ignores NaN
            const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(v));   // order-preserving for v >= 0
            if (lane == 0 && top) atomicMax(&a.maxbits[g], top);
        }
        if (!grid_barrier(a.barrier, target, a.status, a.wait)) return false;
    }

    // ---- flag
    float pool_max = 0.f;
    int max_of = -1;   // the GP that it belongs to
    for (int s = blockIdx.x; s < chunks; s += gridDim.x) {
        const int g = s / a.chunks_per_gp;
        if (a.tile_max && g != max_of) {   // every block takes the largest of the tiles' largest by itself
            float v = 0.f;
#pragma unroll 4
            for (int i = t; i < a.tiles_per_gp; i += kThreads) {
                const float4 q = __ldg(a.tile_max + (size_t)g * a.tiles_per_gp + i);
                v = fmaxf(fmaxf(v, fmaxf(q.x, q.y)), fmaxf(q.z, q.w));
            }
            const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
            __syncthreads();
            if (lane == 0) warp_sum[warp] = (int)top;
            __syncthreads();
            for (int w = 0; w < 8; ++w) pool_max = w ? fmaxf(pool_max, __int_as_float(warp_sum[w])) : __int_as_float(warp_sum[0]);
            max_of = g;
        }
        const long long c0 = (long long)(s % a.chunks_per_gp) * a.chunk, c1 = min(m, c0 + a.chunk);
        const float sf2 = a.sf2v[g], best = a.bestv[g];
        const float tol_ei = 1e-5f * (a.tile_max ? pool_max : __uint_as_float(__ldcg(a.maxbits + g)));
        const float mu_floor = 1e-6f * a.yabsv[g], sd_floor = 1e-6f * sqrtf(sf2);
        if (own_rescue) {
            __syncthreads();
            if (t == 0) own_count = 0;
            __syncthreads();
        }
        constexpr int kBatch = 4;   // loads of so many candidates per thread are under way at a time
        for (long long b0 = c0; b0 < c1; b0 += kBatch * kThreads) {
            float mu4[kBatch], sd4[kBatch], dmu4[kBatch], dq4[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                if (b0 + j * kThreads >= c1) continue;   // the same for the whole block
                const long long i = b0 + j * kThreads + t;
                const size_t f = (size_t)g * m + (i < c1 ? i : c0);
                mu4[j] = __ldcs(a.mu + f);
                sd4[j] = __ldcs(a.sigma + f);
                dmu4[j] = __ldcs(a.err_mu + f);
                dq4[j] = __ldcs(a.err_q + f);
            }
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                if (b0 + j * kThreads >= c1) continue;
                const long long i = b0 + j * kThreads + t;
                const bool flag = i < c1 && misses_contract(mu4[j], sd4[j], dmu4[j], dq4[j], tol_ei, mu_floor, sd_floor, best, sf2);
                const unsigned votes = __ballot_sync(0xffffffffu, flag);   // one counter update per warp
                if (votes) {
                    const int rank = __popc(votes & ((1u << lane) - 1u)), all = __popc(votes);
                    int mine = 0, base = 0;   // the first `mine` of the warp's go to the block's own list
                    if (lane == 0) {
                        atomicAdd(&a.total[g], all);
                        if (own_rescue) {
                            base = atomicAdd(&own_count, all);
                            mine = max(0, min(all, kSmallTile - base));
                        }
                    }
                    if (own_rescue) {
                        base = __shfl_sync(0xffffffffu, base, 0);
                        mine = __shfl_sync(0xffffffffu, mine, 0);
                        if (flag && rank < mine) own[base + rank] = (int)i;
                    }
                    if (mine < all) {
                        if (lane == 0) base = atomicAdd(&a.count[g], all - mine);
                        base = __shfl_sync(0xffffffffu, base, 0);
                        if (flag && rank >= mine) a.list[(size_t)g * m + R3_IDX(base + rank - mine, m, a.status)] = (int)i;
                    }
                }
            }
        }
        if (own_rescue) {
            __syncthreads();
            if (own_count > 0) rescue_own(a, g, own, min(own_count, kSmallTile), smem);
        }
    }
    if (!grid_barrier(a.barrier, target, a.status, a.wait)) return false;
    if (blockIdx.x == 0 && t < min(a.batch, 64)) a.rescued_h[t] = __ldcg(a.total + t);   // pinned host memory

    // ---- rescue
    {
        int* pref = reinterpret_cast<int*>(smem + a.pref_offset);   // [batch + 1] tiles before each GP
        auto prefix = [&](int ct) {
            const int per = (a.batch + kThreads - 1) / kThreads, g0 = t * per, g1 = min(a.batch, g0 + per);
            int mine = 0;
            for (int g = g0; g < g1; ++g) mine += (__ldcg(a.count + g) + ct - 1) / ct;
            int incl = mine;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            __syncthreads();
            if (lane == 31) warp_sum[warp] = incl;
            __syncthreads();
            int before = incl - mine;
            for (int w = 0; w < warp; ++w) before += warp_sum[w];
            for (int g = g0; g < g1; ++g) {
                pref[g] = before;
                before += (__ldcg(a.count + g) + ct - 1) / ct;
            }
            if (g1 == a.batch && g0 < g1) pref[a.batch] = before;
            __syncthreads();
            return pref[a.batch];
        };
        const int big = prefix(kTile);
        if (big > 0) {
            // 64 x 64 tiles once they give every block two; below that 16 x 16 tiles spread the work
            const long long items = (long long)big * ((a.npad + kTile - 1) / kTile);
            if (items >= 2ll * gridDim.x) {
                if (!rescue<kTile>(a, pref, big, target, smem)) return false;
            } else {
                const int small = prefix(kSmallTile);
                if (!rescue<kSmallTile>(a, pref, small, target, smem)) return false;
            }
            if (a.k > 0 && !grid_barrier(a.barrier, target, a.status, a.wait)) return false;
        }
    }
    if (a.k == 0) return true;

    // ---- the k largest final EI of every slice
    unsigned long long* keys_s = reinterpret_cast<unsigned long long*>(smem);
    for (int s = blockIdx.x; s < slices; s += gridDim.x) {
        const int g = s / a.slices_per_gp;
        const long long c0 = (long long)(s % a.slices_per_gp) * a.slice;
        const float* e = a.ei + (size_t)g * m;
        __syncthreads();
#pragma unroll 1
        for (int i0 = t; i0 < a.slice; i0 += 8 * kThreads) {   // eight loads under way at a time
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = i0 + j * kThreads;
                v[j] = i < a.slice && c0 + i < m ? __ldcg(e + c0 + i) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = i0 + j * kThreads;
                if (i < a.slice) keys_s[i] = c0 + i < m ? topk_make_key(v[j], (unsigned)(c0 + i)) : 0ull;
            }
        }
        block_select_desc(keys_s, a.slice, a.K2, smem + a.select_offset);
        unsigned long long* out = a.keys + (size_t)s * a.K2;
        for (int i = t; i < a.K2; i += kThreads) out[i] = keys_s[R3_IDX(i, a.slice, a.status)];
        if (a.finish) {
            __threadfence();
            __syncthreads();
            if (t == 0) last_slice = atomicAdd(&a.done[g], 1u) == (unsigned)a.slices_per_gp - 1u;
            __syncthreads();
            if (last_slice) {   // this block saw the GP's last slice: its keys are all there
                __threadfence();
                const int nk = a.slices_per_gp * a.K2;
                const unsigned long long* in = a.keys + (size_t)g * nk;
#pragma unroll 8
                for (int i = t; i < nk; i += kThreads) keys_s[i] = __ldcg(in + i);
                block_select_desc(keys_s, nk, a.k, smem + a.select_offset);
                for (int i = t; i < a.k; i += kThreads) {
                    const unsigned c = topk_key_index(keys_s[i]);
                    a.idx[(size_t)g * a.k + i] = (int)c;
                    if (a.val) a.val[(size_t)g * a.k + i] = ((long long)c < m) ? __ldcg(e + c) : __int_as_float(0x7fc00000);
                }
            }
        }
    }
    return true;
}

__global__ void __launch_bounds__(kThreads, 2) guard_kernel(const GuardArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if (guard_pool(a, smem) || a.k == 0) return;
    // The results are invalid, and the status word says so, but whoever reads the pool through the selected indices before the
    // status has been looked at must find k different rows of it.
    __syncthreads();
    if (a.finish) {
        for (int e = threadIdx.x; e < a.batch * a.k; e += kThreads) a.idx[e] = e % a.k;
    } else {   // the later levels read these keys
        for (int s = blockIdx.x; s < a.slices_per_gp * a.batch; s += gridDim.x) {
            const long long c0 = (long long)(s % a.slices_per_gp) * a.slice;
            for (int i = threadIdx.x; i < a.K2; i += kThreads)
                a.keys[R3_IDX((size_t)s * a.K2 + i, (size_t)a.slices_per_gp * a.batch * a.K2, a.status)] = c0 + i < a.m ? topk_make_key(0.f, (unsigned)(c0 + i)) : 0ull;
        }
    }
}

// candidates whose FP64 cross-covariances are in the workspace at a time
int slab_candidates(const r3_gp* gp, long long m)
{
    const size_t fit = kSlabBytes / (sizeof(double) * (size_t)gp->npad) / kTile * kTile;
    const size_t all = ((size_t)m + kTile - 1) / kTile * kTile * gp->batch;
    return (int)std::max<size_t>(kTile, std::min(fit, all));
}

size_t up16(size_t b) { return (b + 15) & ~(size_t)15; }

}  // namespace

size_t guard_workspace_bytes(const r3_gp* gp, long long m)
{
    const size_t bm = (size_t)gp->batch * m, slab = slab_candidates(gp, m), npad = gp->npad;
    return 3 * up16(bm * sizeof(float)) + up16((4 * (size_t)gp->batch + 2) * sizeof(int)) +
           sizeof(double) * slab * (npad + npad / 16 + (npad + 63) / 64) + 256;
}

GuardBuffers guard_carve(const r3_gp* gp, long long m, void* ws)
{
    GuardBuffers b;
    const size_t bm = up16((size_t)gp->batch * m * sizeof(float));
    char* p = (char*)(((uintptr_t)ws + 15) & ~(uintptr_t)15);
    b.err_mu = (float*)p;
    p += bm;
    b.err_q = (float*)p;
    p += bm;
    b.list = (int*)p;
    p += bm;
    b.count = (int*)p;
    b.total = b.count + gp->batch;
    b.maxbits = (unsigned*)b.total + gp->batch;
    b.done = b.maxbits + gp->batch;
    b.barrier = b.done + gp->batch;
    b.mode = (int*)b.barrier + 1;
    p += up16((4 * (size_t)gp->batch + 2) * sizeof(int));
    const size_t slab = slab_candidates(gp, m), npad = gp->npad;
    b.ks = (double*)p;
    b.qpart = b.ks + slab * npad;
    b.mupart = b.qpart + slab * (npad / 16);
    return b;
}

// Candidates per chunk: enough chunks to fill the GPU on a large pool, small ones on a small pool.
static int guard_chunk(int batch, long long m)
{
    long long s = 128;
    while (s < 4096 && s < m && s * 296 < (long long)batch * m) s <<= 1;
    return (int)s;
}

// Candidates per slice of the selection: a chunk, or more when that brings the slices' keys down to what the kernel
// finishes by itself (262,144 candidates, k = 32: two more launches and 8192 keys 15 us, one block over 8192 keys 25 us).
static int guard_slice(int batch, long long m, int k)
{
    const long long s = guard_chunk(batch, m);
    auto keys = [&](long long v) { return (m + v - 1) / v * std::min<long long>(k, v); };
    long long v = s;
    while (v < 4096 && v < m && keys(v) > kFinishKeys) v <<= 1;
    return (int)(keys(v) <= kFinishKeys ? v : s);
}

size_t guard_topk_workspace_bytes(int batch, long long m, int k)
{
    const int slice = guard_slice(batch, m, k);
    const long long slices = (m + slice - 1) / slice;
    return 2 * (size_t)batch * slices * std::min(k, slice) * sizeof(unsigned long long) + 64;
}

// counts, maxima, finished slices and the grid barrier
int guard_zero_ints(const r3_gp* gp) { return 4 * gp->batch + 1; }

r3_status_t guard_pilot(r3_gp* gp, long long m, long long rows, const GuardBuffers& b, const float* mu, const float* sigma,
                        const float* ei, cudaStream_t stream)
{
    GuardArgs a = {};
    a.sf2v = gp->sf2_d; a.bestv = gp->best_d; a.yabsv = gp->yabs_d;
    a.m = m;
    a.mu = const_cast<float*>(mu); a.sigma = const_cast<float*>(sigma); a.ei = const_cast<float*>(ei);   // only read
    a.err_mu = b.err_mu; a.err_q = b.err_q;
    R3_LAUNCH(pilot_kernel, 1, 1024, 0, stream, a, rows, b.mode, b.count, guard_zero_ints(gp));
    return R3_OK;
}

r3_status_t guard_and_rescue(r3_gp* gp, const float* Xcand, long long m, const GuardBuffers& b, float* mu,
                             float* sigma, float* ei, const float* tile_max, long long tiles_per_gp, bool have_max, cudaStream_t stream)
{
    const int B = gp->batch;
    const TopkRequest req = gp->topk_req;
    gp->topk_req = TopkRequest();
    GuardArgs a;
    a.X = gp->X; a.ell = gp->ell_d; a.sf2v = gp->sf2_d; a.bestv = gp->best_d; a.yabsv = gp->yabs_d; a.Xcand = Xcand;
    a.alpha64 = gp->alpha64; a.W64 = gp->W64;
    a.batch = B; a.n = gp->n; a.d = gp->d; a.npad = gp->npad;
    a.m = m;
    a.chunk = guard_chunk(B, m);
    a.chunks_per_gp = (int)((m + a.chunk - 1) / a.chunk);
    a.slice = guard_slice(B, m, req.k);
    a.slices_per_gp = (int)((m + a.slice - 1) / a.slice);
    a.mu = mu; a.sigma = sigma; a.ei = ei;
    a.err_mu = b.err_mu; a.err_q = b.err_q;
    a.list = b.list;
    a.maxbits = b.maxbits;
    a.count = b.count;
    a.total = b.total;
    a.rescued_h = gp->rescued_h;
    a.done = b.done;
    a.barrier = b.barrier;
    a.status = gp->status_d;
    a.wait = wait_rule(gp, STALL_GUARD);
    a.have_max = have_max || tile_max;
    a.tile_max = reinterpret_cast<const float4*>(tile_max);
    a.tiles_per_gp = (int)tiles_per_gp;
    a.ks = b.ks; a.qpart = b.qpart; a.mupart = b.mupart;
    a.slab = slab_candidates(gp, m);
    a.k = req.k;
    a.K2 = req.k > 0 ? std::min(req.k, a.slice) : 1;
    a.keys = (unsigned long long*)req.ws;
    a.idx = req.idx;
    a.val = req.val;
    const long long keys_per_gp = (long long)a.slices_per_gp * a.K2;
    a.finish = req.k > 0 && keys_per_gp <= kFinishKeys;
    if (req.k > 0 && req.ws_bytes < guard_topk_workspace_bytes(B, m, req.k)) {
        set_error("internal: top-k workspace of the guard too small");
        return R3_ERR_INVALID_ARG;
    }
    // dynamic shared memory: operand stages / slice keys, then the selection's scratch, then the tile prefix
    size_t region = kCrossStageBytes;
    a.select_offset = (unsigned)(sizeof(unsigned long long) * (a.finish ? (size_t)kFinishKeys : (size_t)a.slice));
    if (req.k > 0) region = std::max(region, a.select_offset + topk_select_scratch_bytes(a.finish ? req.k : a.K2));
    a.pref_offset = (unsigned)up16(region);
    const size_t smem = a.pref_offset + sizeof(int) * ((size_t)B + 1);
    int sms = 148;
    R3_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, gp->device));
    // the cap belongs to the kernel, not to the call: always the most that any call asks for
    R3_CUDA_TRY(cudaFuncSetAttribute(guard_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
    // two blocks per SM (launch bounds and 112 KB of shared memory allow it); a small pool is served by half of them,
    // because the barriers then cost more than the work between them
    const long long chunks = (long long)a.chunks_per_gp * B;
    const unsigned grid = (unsigned)(chunks <= sms ? sms : 2 * sms);
    void* params[] = {&a};
    R3_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)guard_kernel, dim3(grid), dim3(kThreads), params, smem, stream));
    ++g_launches;
    if (req.k == 0 || a.finish) return R3_OK;
    unsigned long long* keys = (unsigned long long*)req.ws;
    return topk_finish_from_keys(keys, keys + (size_t)B * keys_per_gp, B, keys_per_gp, req.k, ei, m, req.idx, req.val, stream);
}

}  // namespace r3
