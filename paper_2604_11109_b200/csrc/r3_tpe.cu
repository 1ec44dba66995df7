// Tree-structured Parzen Estimator: fit (order of the history, per-dimension mixtures and level
// tables) and candidate scoring (log-density ratio), steps (T1)-(T4) of the definition in r3.h.
//
// Fit is small (n <= 4096): one block sorts the history by y, then one block per dimension sorts each
// set's values (bitonic network in shared memory), derives the bandwidths from the neighbour gaps in
// FP64 and stores every component as {mean, a, b, sigma} with
//     a = log2(e) / (2 sigma^2),   b = log2( weight / (sum of weights * sigma * Z * sqrt(2 pi)) ),
// so that the scoring kernel evaluates a component as exp2(b - a (x - mean)^2): one subtraction, one
// multiplication, one fused multiply-add, one MUFU.EX2 and one addition per (candidate, component).
// Scoring is bound by the MUFU unit (16 results per clock per SM); the components of a dimension are
// staged through shared memory and every thread carries one or two candidates.
#include <math.h>
#include <stdlib.h>

#include <algorithm>
#include <new>
#include <vector>

#include "r3_f32x2.cuh"
#include "r3_internal.cuh"

struct r3_tpe {
    int n = 0, d = 0, n_good = 0, device = 0;
    float prior_weight = 1.f;
    std::vector<int> levels;
    int tabled = 0;            // features with a table
    int* levels_d = nullptr;   // [d], then [d]: the features with a table, then those with mixtures (a score adds them up so)
    int* order_d = nullptr;    // [n] history indices by y ascending
    float4* comps_d = nullptr; // [d][n + 2]: good set's components from 0, the bad set's from n_good + 1
    int* counts_d = nullptr;   // [d][2]: components of each set after merging equal ones
    // a model small enough for shared memory is also kept packed: set (j, s) at [offs[2j + s], offs[2j + s + 1])
    int total = 0;             // components kept over all dimensions and sets
    bool resident = false;     // the packed model is in use
    float4* packed_d = nullptr;
    int* offs_d = nullptr;     // [2d + 1]
    char* arena_d = nullptr;   // the one allocation all device pointers of the handle point into
    float* table_d = nullptr;  // [d][64] ln P_good - ln P_bad per level
    int* status_d = nullptr;   // status bits
    int* status_h = nullptr;   // pinned mirror
};

namespace r3 {

namespace {

constexpr int kTpeMaxN = 4096;
constexpr int kTpeMaxLevels = 64;
constexpr int kSortThreads = 1024;
constexpr int kScoreThreads = 256;
constexpr int kStage = 512;   // components per shared-memory stage
constexpr size_t kResidentBytes = 72 * 1024;   // largest model a scoring block keeps whole in shared memory
// Components of such a model with every set padded to a multiple of four: set i begins at its unpadded place plus 3 i, rounded
// up to a multiple of four, which leaves room for the padding of the sets before it.
__host__ __device__ inline int resident_padded(int total, int d) { return (total + 3 * 2 * d + 3) & ~3; }

// Unsigned integer with the same order as the float (-0 and +0 equal).
__device__ __forceinline__ unsigned ordered_bits(float v)
{
    if (v == 0.0f) v = 0.0f;
    const unsigned u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_ordered_bits(unsigned u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

// Ascending bitonic sort of `count` (a power of two, at most 8 blockDim.x) 64-bit keys in shared memory; all threads of the
// block call it.  A warp takes 128 neighbouring keys into registers, four per lane, and makes all steps of distance below
// 128 there, by shuffles and within the lane; the longer distances go through shared memory.
constexpr int kWarpKeys = 128;
__device__ __forceinline__ void order_pair(unsigned long long& a, unsigned long long& b, bool asc)
{
    const bool swap = (a > b) == asc;
    const unsigned long long lo = swap ? b : a, hi = swap ? a : b;
    a = lo;
    b = hi;
}
// Steps of distance `top` (at most 64) and below of the merge to blocks of `size`, for the 128 keys from `first` on.  Lane l
// holds keys first + l + 32 e.
__device__ __forceinline__ void warp_merge(unsigned long long (&k)[4], int first, int size, int top)
{
    const int lane = threadIdx.x & 31;
    const bool asc_all = (first & size) == 0;   // size >= 128: one direction for the whole warp
    for (int stride = top; stride > 0; stride >>= 1) {
        if (stride >= 32) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int o = e ^ (stride >> 5);
                if (o > e) {
                    // (e is a compile-time constant, o one of two: both cases are spelt out by the unrolling)
                    const bool asc = size >= kWarpKeys ? asc_all : ((e * 32) & size) == 0;
                    if (stride == 64) { if (e < 2) order_pair(k[e], k[e + 2], asc); }
                    else if ((e & 1) == 0) order_pair(k[e], k[e + 1], asc);
                }
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int pos = e * 32 + lane;
                const bool asc = size >= kWarpKeys ? asc_all : (pos & size) == 0;
                const unsigned long long other = __shfl_xor_sync(0xffffffffu, k[e], stride);
                const bool low = (lane & stride) == 0;   // this lane keeps the smaller one if ascending
                const bool take = (low == asc) ? other < k[e] : other > k[e];
                k[e] = take ? other : k[e];
            }
        }
    }
}
__device__ __forceinline__ void bitonic_sort_asc(unsigned long long* s, int count)
{
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31, warps = blockDim.x / 32;
    __syncthreads();
    if (count < kWarpKeys) {
        // a handful of keys: one warp, filled up with keys that sort last
        if (warp == 0) {
            unsigned long long k[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) k[e] = e * 32 + lane < count ? s[e * 32 + lane] : ~0ull;
            for (int size = 2; size <= kWarpKeys; size <<= 1) warp_merge(k, 0, size, size >> 1);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (e * 32 + lane < count) s[e * 32 + lane] = k[e];
        }
        __syncthreads();
        return;
    }
    for (int size = kWarpKeys; size <= count; size <<= 1) {
        for (int stride = size >> 1; stride >= kWarpKeys; stride >>= 1) {
            for (int t = threadIdx.x; t < count / 2; t += blockDim.x) {
                const int lo = 2 * t - (t & (stride - 1));
                const int hi = lo + stride;
                const bool asc = ((lo & size) == 0);
                const unsigned long long a = s[lo], b = s[hi];
                if ((a > b) == asc) {
                    s[lo] = b;
                    s[hi] = a;
                }
            }
            __syncthreads();
        }
        for (int first = warp * kWarpKeys; first < count; first += warps * kWarpKeys) {
            unsigned long long k[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) k[e] = s[first + e * 32 + lane];
            if (size == kWarpKeys)
                for (int sz = 2; sz < kWarpKeys; sz <<= 1) warp_merge(k, first, sz, sz >> 1);
            warp_merge(k, first, size, kWarpKeys / 2);
#pragma unroll
            for (int e = 0; e < 4; ++e) s[first + e * 32 + lane] = k[e];
        }
        __syncthreads();
    }
}

__device__ __forceinline__ int pow2_at_least(int v)
{
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// (T1) order[i] = index of the i-th smallest y, ties by lower index: every value counts the ones before it.  n^2 comparisons
// spread over the GPU, kOrderRows values per block, a warp per value, against all of y in shared memory (a sort by one block
// took 40 us for 4096 values; 15 us).
constexpr int kOrderRows = 32;
__global__ void __launch_bounds__(256) tpe_order_kernel(const float* __restrict__ y, int n, int* __restrict__ order,
                                                        int* __restrict__ status)
{
    __shared__ unsigned bits[kTpeMaxN];
    bool bad = false;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float v = y[i];
        bad |= !isfinite(v);
        bits[i] = ordered_bits(v);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, DEV_NONFINITE);
    const int lane = threadIdx.x & 31;
    for (int r = threadIdx.x / 32; r < kOrderRows; r += blockDim.x / 32) {
        const int i = blockIdx.x * kOrderRows + r;
        if (i >= n) break;
        const unsigned mine = bits[i];
        int before = 0;
#pragma unroll 8
        for (int k = lane; k < n; k += 32) before += bits[k] < mine || (bits[k] == mine && k < i) ? 1 : 0;
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane == 0) order[before] = i;
    }
}

// (T2), (T3): one block per (dimension, set).  Bound: the sort.  64 dimensions, 4096 observations, 16 distinct values each:
// 60 us; 737 us while one thread walked the sorted values to merge equal components, all of which had their truncation mass
// computed first.  The log-probabilities (categorical) or log-densities (grid) of a
// set go to lnp[j][set][v]; tpe_table_kernel subtracts the two sets afterwards.
__global__ void __launch_bounds__(kSortThreads) tpe_mixture_kernel(const float* __restrict__ X,
                                                                   const int* __restrict__ order, int n, int d,
                                                                   int n_good, const int* __restrict__ levels,
                                                                   double prior_weight, float4* __restrict__ comps,
                                                                   int* __restrict__ n_comps, double* __restrict__ lnp_out,
                                                                   int* __restrict__ status)
{
    extern __shared__ unsigned long long keys[];   // pow2 >= n + 1 keys, then 3 (n + 2) doubles
    __shared__ int counts[kTpeMaxLevels];
    __shared__ int warp_count[32];
    const int j = blockIdx.x >> 1;
    const int code = levels[j];
    const int C = code > 0 ? code : 0;      // categorical levels
    const int G = code < 0 ? -code : 0;     // grid values of an ordinal dimension
    bool bad = false;
    double* lnp_set = lnp_out + ((size_t)j * 2 + (blockIdx.x & 1)) * kTpeMaxLevels;
    for (int set = blockIdx.x & 1; set == (int)(blockIdx.x & 1); set += 2) {
        const int s = set == 0 ? n_good : n - n_good;
        const int first = set == 0 ? 0 : n_good;            // position in `order`
        float4* out = comps + (size_t)j * (n + 2) + (set == 0 ? 0 : n_good + 1);
        if (C > 0) {
            // ---- (T3) smoothed level frequencies
            for (int v = threadIdx.x; v < kTpeMaxLevels; v += blockDim.x) counts[v] = 0;
            __syncthreads();
            for (int i = threadIdx.x; i < s; i += blockDim.x) {
                const float x = X[(size_t)order[first + i] * d + j];
                bad |= !isfinite(x);
                const float lv = floorf(__fadd_rn(__fmul_rn(x, (float)(C - 1)), 0.5f));
                const int v = (int)fminf(fmaxf(lv, 0.f), (float)(C - 1));
                atomicAdd(&counts[isfinite(x) ? v : 0], 1);
            }
            __syncthreads();
            for (int v = threadIdx.x; v < C; v += blockDim.x) {
                lnp_set[v] = log(((double)counts[v] + prior_weight / C) / ((double)s + prior_weight));
            }
            if (threadIdx.x == 0) n_comps[2 * j + set] = 0;
            __syncthreads();
            continue;
        }
        // ---- (T2) sort the s values and the prior mean; the prior (index s) goes after equal values
        const int count = pow2_at_least(s + 1);
        for (int i = threadIdx.x; i < count; i += blockDim.x) {
            unsigned long long k = ~0ull;
            if (i < s) {
                const float x = X[(size_t)order[first + i] * d + j];
                bad |= !isfinite(x);
                k = ((unsigned long long)ordered_bits(isfinite(x) ? x : 0.f) << 32) | (unsigned)i;
            } else if (i == s) {
                k = ((unsigned long long)ordered_bits(0.5f) << 32) | (unsigned)s;
            }
            keys[i] = k;
        }
        bitonic_sort_asc(keys, count);
        const double sigma_lo = 1.0 / fmin(100.0, (double)s + 1.0);
        const double wsum = (double)s + prior_weight;
        auto mean_bits = [&](int t) { return (unsigned)(keys[t] >> 32); };
        auto mean_of = [&](int t) { return (double)from_ordered_bits(mean_bits(t)); };
        auto sigma_of = [&](int t) {
            if ((int)(keys[t] & 0xFFFFFFFFull) == s) return 1.0;   // the prior
            const double mu = mean_of(t);
            double gap = -1.0;
            if (t > 0) gap = fmax(gap, mu - mean_of(t - 1));
            if (t < s) gap = fmax(gap, mean_of(t + 1) - mu);
            return fmin(fmax(gap, sigma_lo), 1.0);
        };
        // Components with the same mean and bandwidth (repeated values of a discrete feature) are one component with the
        // summed coefficient: the density is the same sum, with far fewer terms.  Equal means are neighbours in the sorted
        // order, and such a run has at most four bandwidths: its first value, the values inside, its last value, the prior.
        // The first value of a run with its bandwidth stands for all of them; every thread finds that out for its own.
        double* comp = reinterpret_cast<double*>(keys + count);   // [c][3]: mean, sigma, coefficient
        int done_before = 0;
        for (int t0 = 0; t0 <= s; t0 += blockDim.x) {
            const int t = t0 + threadIdx.x;
            bool leader = false;
            double sigma = 0.0, coef = 0.0;
            if (t <= s) {
                const unsigned mu_bits = mean_bits(t);
                sigma = sigma_of(t);
                leader = true;
                if (t > 0 && mean_bits(t - 1) == mu_bits) {
                    int lo = 0, hi = t;   // the run's first position
                    while (lo < hi) {
                        const int mid = (lo + hi) / 2;
                        if (mean_bits(mid) < mu_bits) lo = mid + 1;
                        else hi = mid;
                    }
                    leader = sigma_of(lo) != sigma && (lo + 1 >= t || sigma_of(lo + 1) != sigma) && sigma_of(t - 1) != sigma;
                }
                if (leader) {
                    // how many values of the run share the bandwidth, and whether the prior does
                    int lo = t, hi = s + 1;   // one past the run
                    while (lo < hi) {
                        const int mid = (lo + hi) / 2;
                        if (mean_bits(mid) <= mu_bits) lo = mid + 1;
                        else hi = mid;
                    }
                    const int last = lo - 1;
                    const bool with_prior = (int)(keys[last] & 0xFFFFFFFFull) == s;
                    const int last_value = with_prior ? last - 1 : last;
                    double weight = with_prior && sigma == 1.0 ? prior_weight : 0.0;
                    // values t .. last_value: itself, those strictly inside (one bandwidth), the last
                    if (t <= last_value) {
                        weight += 1.0;
                        if (t < last_value) {
                            const int inside = last_value - t - 1;
                            if (inside > 0 && sigma_of(t + 1) == sigma) weight += (double)inside;
                            if (sigma_of(last_value) == sigma) weight += 1.0;
                        }
                    }
                    const double mu = mean_of(t);
                    const double Z = 0.5 * erfc(-(1.0 - mu) / sigma * 0.70710678118654752440) -
                                     0.5 * erfc(-(0.0 - mu) / sigma * 0.70710678118654752440);
                    coef = weight / (wsum * sigma * Z * 2.5066282746310005024);
                }
            }
            // place among the leaders: order of the sorted positions
            const unsigned votes = __ballot_sync(0xffffffffu, leader);
            __syncthreads();
            if ((threadIdx.x & 31) == 0) warp_count[threadIdx.x / 32] = __popc(votes);
            __syncthreads();
            int before = done_before, all = 0;
            for (int w = 0; w < (int)blockDim.x / 32; ++w) {
                if (w < (int)threadIdx.x / 32) before += warp_count[w];
                all += warp_count[w];
            }
            done_before += all;
            if (leader) {
                const int c = before + __popc(votes & ((1u << (threadIdx.x & 31)) - 1u));
                comp[3 * c] = mean_of(t);
                comp[3 * c + 1] = sigma;
                comp[3 * c + 2] = coef;
                const double a = 1.4426950408889634074 / (2.0 * sigma * sigma);
                out[c] = make_float4(from_ordered_bits(mean_bits(t)), (float)a, (float)log2(coef), (float)sigma);
            }
        }
        if (threadIdx.x == 0) n_comps[2 * j + set] = done_before;
        __syncthreads();
        // (T3g) the mixture at each of the G grid values, in FP64, a warp per value
        for (int v = threadIdx.x / 32; v < G; v += blockDim.x / 32) {
            const double xg = (double)(float)((double)v / (double)(G - 1));
            double acc = 0.0;
            for (int c = threadIdx.x & 31; c < done_before; c += 32) {
                const double z = (xg - comp[3 * c]) / comp[3 * c + 1];
                acc += comp[3 * c + 2] * exp(-0.5 * z * z);
            }
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if ((threadIdx.x & 31) == 0) lnp_set[v] = log(acc);
        }
    }
    if (bad) atomicOr(status, DEV_NONFINITE);
}

// (T3), (T3g): table[j][v] = ln l_j(v) - ln g_j(v) for the tabulated dimensions, zero elsewhere
__global__ void tpe_table_kernel(const int* __restrict__ levels, const double* __restrict__ lnp, int d,
                                 float* __restrict__ table)
{
    const int j = blockIdx.x, v = threadIdx.x;
    const int code = levels[j];
    const int cnt = code < 0 ? -code : code;
    const double* l = lnp + (size_t)j * 2 * kTpeMaxLevels;
    table[(size_t)j * kTpeMaxLevels + v] = v < cnt ? (float)(l[v] - l[kTpeMaxLevels + v]) : 0.f;
}

__device__ __forceinline__ float ex2_fast(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float lg2_fast(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Components in shared memory, one array per coefficient: -mean, -a and b of four components in a row are three 16-byte reads
// and give two pairs of each, ready for the packed FP32 instructions.  Sets are padded to a multiple of four with components
// that contribute nothing.
struct Components {
    float *nmean, *na, *b;
};
constexpr float kNullB = -1e4f;   // exp2 of it is 0 either way

__device__ __forceinline__ uint64_t both(float v) { return pack2(v, v); }

// exp2 of a pair on the FP32 pipe: x = n + f with n the nearest whole number, 2^f by a polynomial ((2^f - 1) / f interpolated at
// six Chebyshev nodes of [-1/2, 1/2]; 7.4e-8 relative at most, the special-function unit 1.7e-7), n added to the exponent.
// Below -127 the result is 0 (n = -127, f = 0), between -127 and -126 less than 2^-126.  x must be below 127.
__device__ __forceinline__ uint64_t exp2_poly2(uint64_t x2)
{
    float x0, x1;
    unpack2(x2, x0, x1);
    x2 = pack2(fmaxf(x0, -127.f), fmaxf(x1, -127.f));
    const uint64_t z = add2(x2, both(12582912.f));           // 1.5 * 2^23: the low bits of z are n
    const uint64_t n = add2(z, both(-12582912.f));
    const uint64_t f = fma2(n, both(-1.f), x2);
    uint64_t p = both(0x1.44138ap-13f);
    p = fma2(p, f, both(0x1.5f0890p-10f));
    p = fma2(p, f, both(0x1.3b2a54p-7f));
    p = fma2(p, f, both(0x1.c6af6cp-5f));
    p = fma2(p, f, both(0x1.ebfbe0p-3f));
    p = fma2(p, f, both(0x1.62e430p-1f));
    p = fma2(p, f, both(1.f));
    float z0, z1, p0, p1;
    unpack2(z, z0, z1);
    unpack2(p, p0, p1);
    return pack2(__int_as_float(__float_as_int(p0) + (__float_as_int(z0) << 23)),
                 __int_as_float(__float_as_int(p1) + (__float_as_int(z1) << 23)));
}
__device__ __forceinline__ uint64_t exp2_fast2(uint64_t x2)
{
    float x0, x1;
    unpack2(x2, x0, x1);
    return pack2(ex2_fast(x0), ex2_fast(x1));
}

// sum over components [lo, hi) (multiples of four) of exp2(b - a (x - mean)^2) for R candidates at once, four partial sums per
// candidate.  Bound by the special-function unit, which gives a warp an exponential in eight cycles, and by instruction issue;
// hence pairs, and with two candidates per thread one exponential in eight on the FP32 pipe.  1,048,576 candidates with 2432
// exponentials each (whole call) and 500,000 with 20,000: scalar instructions 1.02 and 2.79 ms, pairs 0.95 and 2.59 ms, one in
// four on the FP32 pipe 0.96 and 2.58 ms, one in eight 0.925 and 2.39 ms.
template <int R>
__device__ __forceinline__ void mixture_sums(const Components& m, int lo, int hi, const float (&x)[R], uint64_t (&part)[R][2])
{
    uint64_t x2[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x2[r] = both(x[r]);
    auto group = [&](int c, bool odd) {
        const ulonglong2 nm = *reinterpret_cast<const ulonglong2*>(m.nmean + c);
        const ulonglong2 na = *reinterpret_cast<const ulonglong2*>(m.na + c);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(m.b + c);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint64_t t0 = add2(x2[r], nm.x), t1 = add2(x2[r], nm.y);
            const uint64_t e0 = fma2(t0, mul2(t0, na.x), b.x), e1 = fma2(t1, mul2(t1, na.y), b.y);
            part[r][0] = add2(part[r][0], exp2_fast2(e0));
            part[r][1] = add2(part[r][1], (r % 2 == 1 && odd) ? exp2_poly2(e1) : exp2_fast2(e1));
        }
    };
    int c = lo;
#pragma unroll 2
    for (; c + 8 <= hi; c += 8) {
        group(c, false);
        group(c + 4, true);
    }
    if (c < hi) group(c, false);
}
template <int R>
__device__ __forceinline__ void finish_sums(const uint64_t (&part)[R][2], float (&sum)[R])
{
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float a, b;
        unpack2(add2(part[r][0], part[r][1]), a, b);
        sum[r] = a + b;
    }
}

// The same over `count` components in global memory, which the whole block stages through shared memory (all of its threads
// must call this together): one broadcast read instead of a global load per thread was worth 14 % on the full pool.
template <int R>
__device__ __forceinline__ void mixture_sums_staged(const float4* __restrict__ comp, int count, const float (&x)[R],
                                                    float (&sum)[R], const Components& stage)
{
    uint64_t part[R][2] = {};
    for (int c0 = 0; c0 < count; c0 += kStage) {
        const int nc = min(kStage, count - c0), nc4 = (nc + 3) & ~3;
        __syncthreads();
        for (int i = threadIdx.x; i < nc4; i += kScoreThreads) {
            const float4 q = i < nc ? __ldg(comp + c0 + i) : make_float4(0.f, 1.f, kNullB, 0.f);
            stage.nmean[i] = -q.x;
            stage.na[i] = -q.y;
            stage.b[i] = q.z;
        }
        __syncthreads();
        mixture_sums<R>(stage, 0, nc4, x, part);
    }
    finish_sums<R>(part, sum);
}

// Look-ups of tabulated features do not depend on one another: in a loop of their own they are taken in groups of four, with the
// next group's values on their way meanwhile, while in one loop with the mixtures each feature waits for the one before it.
// Bound by the latency of those reads.  400,000 candidates with 59 tables and a mixture of 40 observations 117 us in one loop,
// 70 us in two.
struct Features {
    int at[kMaxD];      // tables first: the features with a table, then those with mixtures; otherwise feature i
    float top[kMaxD];   // admissible values - 1, -1 for a mixture
};
template <bool TABLES_FIRST>
__device__ __forceinline__ void load_features(Features& s, const int* __restrict__ levels, int d)
{
    for (int i = threadIdx.x; i < d; i += kScoreThreads) {
        s.at[i] = TABLES_FIRST ? __ldg(levels + d + i) : i;
        s.top[i] = (float)(abs(__ldg(levels + s.at[i])) - 1);
    }
}
// the admissible value nearest to x (top + 1 of them)
__device__ __forceinline__ int level_of(float x, float top)
{
    const float lv = floorf(__fadd_rn(__fmul_rn(x, top), 0.5f));
    return isfinite(x) ? (int)fminf(fmaxf(lv, 0.f), top) : 0;
}
// acc[r] += the tables' contributions to the candidate in row[r] (a row of the pool for every r)
template <int R>
__device__ __forceinline__ void add_tabled(const Features& s, int tabled, const float* const (&row)[R], const float* __restrict__ table,
                                           float (&acc)[R], bool& bad)
{
    if (tabled == 0) return;
    float next[R][4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int r = 0; r < R; ++r) next[r][e] = e < tabled ? row[r][s.at[e]] : 0.f;
    for (int i0 = 0; i0 < tabled; i0 += 4) {
        float x[R][4], found[R][4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                x[r][e] = next[r][e];
                next[r][e] = i0 + 4 + e < tabled ? row[r][s.at[i0 + 4 + e]] : 0.f;
            }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (i0 + e >= tabled) continue;
            const float top = s.top[i0 + e];
            const float* t = table + (size_t)s.at[i0 + e] * kTpeMaxLevels;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                bad |= !isfinite(x[r][e]);
                found[r][e] = __ldg(t + level_of(x[r][e], top));
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (i0 + e < tabled) acc[r] += found[r][e];
    }
}

// (T4) score of every candidate.  A block covers R * blockDim.x consecutive candidates; thread t holds
// candidates t, t + blockDim.x, ... of the block's range so that the result stores coalesce.
template <int R>
__global__ void __launch_bounds__(kScoreThreads) tpe_score_kernel(const float* __restrict__ Xc, long long m, int n,
                                                                  int d, int n_good, const int* __restrict__ levels, int tabled,
                                                                  const float4* __restrict__ comps,
                                                                  const int* __restrict__ counts,
                                                                  const float* __restrict__ table,
                                                                  float* __restrict__ score, int* __restrict__ status)
{
    const long long tiles = (m + (long long)R * kScoreThreads - 1) / ((long long)R * kScoreThreads);
    bool bad = false;
    __shared__ __align__(16) float stage_s[3][kStage];
    const Components stage{stage_s[0], stage_s[1], stage_s[2]};
    constexpr bool SPLIT = R == 1;   // the tables in a loop of their own (3000 candidates, 98 tables and two mixtures: 172 -> 135 us)
    __shared__ Features features;
    if constexpr (SPLIT) {
        load_features<true>(features, levels, d);
        __syncthreads();
    }
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long base = tile * (long long)R * kScoreThreads + threadIdx.x;
        const float* row[R];
        bool valid[R];
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long cand = base + (long long)r * kScoreThreads;
            valid[r] = cand < m;
            row[r] = Xc + (size_t)(valid[r] ? cand : 0) * d;
            acc[r] = 0.f;
        }
        if constexpr (SPLIT) add_tabled<R>(features, tabled, row, table, acc, bad);
        for (int i = SPLIT ? tabled : 0; i < d; ++i) {
            const int j = SPLIT ? features.at[i] : i;
            float x[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                x[r] = row[r][j];
                bad |= valid[r] && !isfinite(x[r]);
            }
            if constexpr (!SPLIT) {
                const int values = abs(__ldg(levels + j));
                if (values > 0) {
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        acc[r] += __ldg(table + (size_t)j * kTpeMaxLevels + level_of(x[r], (float)(values - 1)));
                    continue;
                }
            }
            const float4* cj = comps + (size_t)j * (n + 2);
            float sl[R], sg[R];
            mixture_sums_staged<R>(cj, __ldg(counts + 2 * j), x, sl, stage);
            mixture_sums_staged<R>(cj + n_good + 1, __ldg(counts + 2 * j + 1), x, sg, stage);
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] += 0.69314718f * (lg2_fast(sl[r]) - lg2_fast(sg[r]));
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (valid[r]) score[base + (long long)r * kScoreThreads] = acc[r];
    }
    if (bad) atomicOr(status, DEV_NONFINITE);
}

// One (dimension, set) per block: where its kept components begin in the packed model, and, if the whole model fits
// `limit` components, their copy there.
__global__ void __launch_bounds__(256) tpe_pack_kernel(const float4* __restrict__ comps, const int* __restrict__ counts, int n,
                                                       int n_good, int sets, int limit, int* __restrict__ offs,
                                                       float4* __restrict__ packed)
{
    __shared__ int sums[2];
    const int b = blockIdx.x, j = b >> 1, set = b & 1;
    if (threadIdx.x < 2) sums[threadIdx.x] = 0;
    __syncthreads();
    int before = 0, all = 0;
    for (int i = threadIdx.x; i < sets; i += blockDim.x) {
        const int c = counts[i];
        all += c;
        if (i < b) before += c;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    all = __reduce_add_sync(0xffffffffu, all);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&sums[0], before);
        atomicAdd(&sums[1], all);
    }
    __syncthreads();
    const int lo = sums[0], cnt = counts[b];
    if (threadIdx.x == 0) {
        offs[b] = lo;
        if (b == sets - 1) offs[sets] = sums[1];
    }
    if (sums[1] > limit) return;
    const float4* src = comps + (size_t)j * (n + 2) + (set ? n_good + 1 : 0);
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) packed[lo + i] = src[i];
}

// (T4) for a model that fits shared memory (discrete features leave a few components per admissible value):
// every block loads the packed model once and then walks its tiles without a block-wide barrier.  (Reading
// four or eight features of a row per load, with the feature loop unrolled to match, measured 10-30 % slower:
// the kernel is bound by instruction issue, not by the row reads.)
// SPLIT: the tables in a loop of their own, behind the mixtures.  It takes more registers and instructions than a branch in one
// loop, which with two candidates per thread only a model of mostly tables pays back (1,048,576 candidates: 59 tables and a
// mixture 215 -> 141 us, five and one 33.7 -> 35.7 us, 32 and 32 695 -> 735 us); with one per thread the reads' latency counts
// for more (60,000 candidates, 32 and 32: 69 -> 62 us).
template <int R, bool SPLIT>
__global__ void __launch_bounds__(kScoreThreads) tpe_score_resident_kernel(
    const float* __restrict__ Xc, long long m, int d, const int* __restrict__ levels, int tabled, const int* __restrict__ offs,
    const float4* __restrict__ packed, int total, const float* __restrict__ table, float* __restrict__ score,
    int* __restrict__ status)
{
    // three arrays of padded components, the features of the mixture loop and where their two sets begin and end, [2d + 1] offsets
    extern __shared__ __align__(16) float model[];
    __shared__ Features features;
    const int padded = resident_padded(total, d);
    const Components comps{model, model + padded, model + 2 * padded};
    const int first = SPLIT ? tabled : 0;
    int4* sets = reinterpret_cast<int4*>(model + 3 * padded);   // padded is a multiple of four
    int* offs_s = reinterpret_cast<int*>(sets + d - first);
    for (int i = threadIdx.x; i <= 2 * d; i += kScoreThreads) offs_s[i] = __ldg(offs + i);
    load_features<SPLIT>(features, levels, d);
    for (int i = threadIdx.x; i < padded; i += kScoreThreads) {
        comps.nmean[i] = 0.f;
        comps.na[i] = -1.f;
        comps.b[i] = kNullB;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < total; c += kScoreThreads) {
        const float4 q = __ldg(packed + c);
        int lo = 0, hi = 2 * d - 1;   // the last set that begins at or before c
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (offs_s[mid] <= c) lo = mid;
            else hi = mid - 1;
        }
        const int at = ((offs_s[lo] + 3 * lo + 3) & ~3) + c - offs_s[lo];
        comps.nmean[at] = -q.x;
        comps.na[at] = -q.y;
        comps.b[at] = q.z;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < d - first; i += kScoreThreads) {
        const int j = features.at[first + i];
        auto padded_at = [&](int set) { return (offs_s[set] + 3 * set + 3) & ~3; };
        sets[i] = make_int4(j, padded_at(2 * j), padded_at(2 * j + 1), padded_at(2 * j + 2));
    }
    __syncthreads();
    const long long tiles = (m + (long long)R * kScoreThreads - 1) / ((long long)R * kScoreThreads);
    bool bad = false;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long base = tile * (long long)R * kScoreThreads + threadIdx.x;
        const float* row[R];
        bool valid[R];
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long cand = base + (long long)r * kScoreThreads;
            valid[r] = cand < m;
            row[r] = Xc + (size_t)(valid[r] ? cand : 0) * d;
            acc[r] = 0.f;
        }
        for (int i = 0; i < d - first; ++i) {
            const int4 q = sets[i];
            float x[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                x[r] = row[r][SPLIT ? q.x : i];
                bad |= valid[r] && !isfinite(x[r]);
            }
            if (!SPLIT && features.top[i] >= 0.f) {
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] += __ldg(table + (size_t)i * kTpeMaxLevels + level_of(x[r], features.top[i]));
                continue;
            }
            float sl[R], sg[R];
            uint64_t part[R][2] = {};
            mixture_sums<R>(comps, q.y, q.z, x, part);
            finish_sums<R>(part, sl);
#pragma unroll
            for (int r = 0; r < R; ++r) part[r][0] = part[r][1] = 0;
            mixture_sums<R>(comps, q.z, q.w, x, part);
            finish_sums<R>(part, sg);
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] += 0.69314718f * (lg2_fast(sl[r]) - lg2_fast(sg[r]));
        }
        if (SPLIT) add_tabled<R>(features, tabled, row, table, acc, bad);
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (valid[r]) score[base + (long long)r * kScoreThreads] = acc[r];
    }
    if (bad) atomicOr(status, DEV_NONFINITE);
}

// (T4) when every dimension is tabulated (categorical or grid) and d is a multiple of 4: the score is
// d look-ups per candidate and the kernel is a streaming read of the pool.  LPC lanes share a candidate
// (each takes every LPC-th group of four features, a 16-byte load), so that a warp reads whole rows
// contiguously; their partial sums meet by shuffles.  A lane always serves the same features, so the block
// keeps a copy of the tables laid out by lane -- entry (iteration, feature-in-group, level) of lane l at
// word ((it*4 + e)*64 + level)*32 + l -- which makes every look-up conflict-free.  Four candidates per
// lane group are in flight.
template <int LPC>
__global__ void __launch_bounds__(256) tpe_table_score_kernel(const float* __restrict__ Xc, long long m, int d,
                                                              const int* __restrict__ levels,
                                                              const float* __restrict__ table,
                                                              float* __restrict__ score, int* __restrict__ status)
{
    constexpr int CPW = 32 / LPC;          // candidates per warp and step
    constexpr int UNROLL = 4;
    extern __shared__ float tsm[];         // [iters][4][64][32] tables by lane, then [iters][4][32] level scales
    const int d4 = d / 4;
    const int iters = (d4 + LPC - 1) / LPC;
    float* scale_sm = tsm + (size_t)iters * 4 * kTpeMaxLevels * 32;
    for (int w = threadIdx.x; w < iters * 4 * kTpeMaxLevels * 32; w += blockDim.x) {
        const int l = w % 32, v = (w / 32) % kTpeMaxLevels, e = (w / (32 * kTpeMaxLevels)) % 4;
        const int it = w / (32 * kTpeMaxLevels * 4);
        const int j4 = l % LPC + it * LPC;
        tsm[w] = j4 < d4 ? table[(size_t)(4 * j4 + e) * kTpeMaxLevels + v] : 0.f;
    }
    for (int w = threadIdx.x; w < iters * 4 * 32; w += blockDim.x) {
        const int l = w % 32, e = (w / 32) % 4, it = w / 128;
        const int j4 = l % LPC + it * LPC;
        const int code = j4 < d4 ? levels[4 * j4 + e] : 2;
        scale_sm[w] = (float)((code < 0 ? -code : code) - 1);
    }
    __syncthreads();
    const int lane = threadIdx.x % 32, sub = lane % LPC;
    const long long warp = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const long long nwarps = (long long)gridDim.x * (blockDim.x / 32);
    bool bad = false;
    for (long long c0 = warp * CPW * UNROLL; c0 < m; c0 += nwarps * CPW * UNROLL) {
        float acc[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) acc[u] = 0.f;
        for (int it = 0; it < iters; ++it) {
            const int j4 = sub + it * LPC;
            float4 x[UNROLL];
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const long long cand = c0 + u * CPW + lane / LPC;
                x[u] = (cand < m && j4 < d4) ? __ldcs(reinterpret_cast<const float4*>(Xc + (size_t)cand * d) + j4)
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float cm1 = scale_sm[(it * 4 + e) * 32 + lane];
                const float* tl = tsm + (size_t)(it * 4 + e) * kTpeMaxLevels * 32 + lane;
#pragma unroll
                for (int u = 0; u < UNROLL; ++u) {
                    const float xe = e == 0 ? x[u].x : (e == 1 ? x[u].y : (e == 2 ? x[u].z : x[u].w));
                    bad |= !isfinite(xe);
                    const float lv = floorf(__fadd_rn(__fmul_rn(xe, cm1), 0.5f));
                    const int v = isfinite(xe) ? (int)fminf(fmaxf(lv, 0.f), cm1) : 0;
                    acc[u] += tl[v * 32];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
#pragma unroll
            for (int o = LPC / 2; o > 0; o >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
            const long long cand = c0 + u * CPW + lane / LPC;
            if (sub == 0 && cand < m) score[cand] = acc[u];
        }
    }
    if (bad) atomicOr(status, DEV_NONFINITE);
}

// (T4) when every dimension is tabulated and rows cannot be read as groups of four (d no multiple of 4, or a pool off a 16-byte
// boundary).  Whatever mixtures the fit kept for a grid are not looked at.  63 features: 2000 candidates 54 us with the kernels
// that have mixtures in mind, 21 us here; 1,000,000 candidates 345 and 121 us.
template <int R>
__global__ void __launch_bounds__(kScoreThreads) tpe_lookup_score_kernel(const float* __restrict__ Xc, long long m, int d,
                                                                         const int* __restrict__ levels,
                                                                         const float* __restrict__ table,
                                                                         float* __restrict__ score, int* __restrict__ status)
{
    __shared__ Features features;
    load_features<true>(features, levels, d);
    __syncthreads();
    const long long tiles = (m + (long long)R * kScoreThreads - 1) / ((long long)R * kScoreThreads);
    bool bad = false;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long base = tile * (long long)R * kScoreThreads + threadIdx.x;
        const float* row[R];
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long cand = base + (long long)r * kScoreThreads;
            row[r] = Xc + (size_t)(cand < m ? cand : 0) * d;
            acc[r] = 0.f;
        }
        add_tabled<R>(features, d, row, table, acc, bad);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long cand = base + (long long)r * kScoreThreads;
            if (cand < m) score[cand] = acc[r];
        }
    }
    if (bad) atomicOr(status, DEV_NONFINITE);
}

size_t resident_bytes(int total, int d) { return sizeof(float4) * (size_t)total + sizeof(int) * (3 * (size_t)d + 1); }

void tpe_destroy(r3_tpe* t)
{
    if (!t) return;
    dev_free(t->arena_d);
    pinned_word_release(t->status_h);
    delete t;
}

r3_status_t tpe_fit_impl(r3_tpe* t, const float* X, const float* y, cudaStream_t stream)
{
    const int n = t->n, d = t->d;
    R3_CUDA_TRY(cudaGetDevice(&t->device));
    // one block of device memory for the whole model (the library's cache hands it back to the next fit)
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t b_comps = up(sizeof(float4) * (size_t)d * (n + 2)), b_packed = up(kResidentBytes),
                 b_table = up(sizeof(float) * (size_t)d * kTpeMaxLevels), b_order = up(sizeof(int) * n),
                 b_levels = up(sizeof(int) * 2 * (size_t)d), b_counts = up(sizeof(int) * 2 * (size_t)d),
                 b_offs = up(sizeof(int) * (2 * (size_t)d + 1)), b_status = 256,
                 b_lnp = up(sizeof(double) * 2 * (size_t)d * kTpeMaxLevels);
    char* base = nullptr;
    if (dev_malloc(&base, b_comps + b_packed + b_table + b_order + b_levels + b_counts + b_offs + b_status + b_lnp) !=
        cudaSuccess) {
        cudaGetLastError();
        set_error("r3_tpe_fit: out of device memory");
        return R3_ERR_ALLOC;
    }
    t->arena_d = base;
    t->comps_d = reinterpret_cast<float4*>(base); base += b_comps;
    t->packed_d = reinterpret_cast<float4*>(base); base += b_packed;
    t->table_d = reinterpret_cast<float*>(base); base += b_table;
    t->order_d = reinterpret_cast<int*>(base); base += b_order;
    t->levels_d = reinterpret_cast<int*>(base); base += b_levels;
    t->counts_d = reinterpret_cast<int*>(base); base += b_counts;
    t->offs_d = reinterpret_cast<int*>(base); base += b_offs;
    t->status_d = reinterpret_cast<int*>(base); base += b_status;
    double* lnp_d = reinterpret_cast<double*>(base);   // scratch of the fit
    t->status_h = pinned_word_acquire();
    if (!t->status_h) {
        set_error("r3_tpe_fit: no pinned host memory");
        return R3_ERR_ALLOC;
    }
    std::vector<int> upload(t->levels);
    for (int tabulated = 1; tabulated >= 0; --tabulated) {
        for (int j = 0; j < d; ++j)
            if ((t->levels[j] != 0) == (tabulated == 1)) upload.push_back(j);
        if (tabulated) t->tabled = (int)upload.size() - d;
    }
    R3_CUDA_TRY(cudaMemcpyAsync(t->levels_d, upload.data(), sizeof(int) * 2 * (size_t)d, cudaMemcpyHostToDevice, stream));
    R3_CUDA_TRY(cudaMemsetAsync(t->status_d, 0, sizeof(int), stream));
    R3_LAUNCH(tpe_order_kernel, (n + kOrderRows - 1) / kOrderRows, 256, 0, stream, y, n, t->order_d, t->status_d);
    int count = 1;
    while (count < n + 1) count <<= 1;
    const size_t smem = sizeof(unsigned long long) * (size_t)count + sizeof(double) * 3 * ((size_t)n + 2);
    if (smem > 48 * 1024)
        R3_CUDA_TRY(cudaFuncSetAttribute(tpe_mixture_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    R3_LAUNCH(tpe_mixture_kernel, 2 * d, kSortThreads, smem, stream, X, t->order_d, n, d, t->n_good, t->levels_d,
              (double)t->prior_weight, t->comps_d, t->counts_d, lnp_d, t->status_d);
    R3_LAUNCH(tpe_table_kernel, d, kTpeMaxLevels, 0, stream, t->levels_d, lnp_d, d, t->table_d);
    // a model that a scoring block can hold in shared memory is packed
    const int limit = (int)((kResidentBytes - resident_bytes(0, d)) / sizeof(float4));
    R3_LAUNCH(tpe_pack_kernel, 2 * d, 256, 0, stream, t->comps_d, t->counts_d, n, t->n_good, 2 * d, limit, t->offs_d, t->packed_d);
    R3_CUDA_TRY(cudaMemcpyAsync(t->status_h, t->status_d, sizeof(int), cudaMemcpyDeviceToHost, stream));
    R3_CUDA_TRY(cudaMemcpyAsync(t->status_h + 1, t->offs_d + 2 * d, sizeof(int), cudaMemcpyDeviceToHost, stream));
    R3_CUDA_TRY(cudaStreamSynchronize(stream));
    if (t->status_h[0] & DEV_NONFINITE) {
        set_error("r3_tpe_fit: X or y contains NaN or Inf");
        return R3_ERR_NONFINITE;
    }
    t->total = t->status_h[1];
    t->resident = t->total > 0 && t->total <= limit;
    return R3_OK;
}

}  // namespace

}  // namespace r3

using namespace r3;

extern "C" {

r3_status_t r3_tpe_fit(const float* X, const float* y, const int* levels, int n, int d, float gamma,
                       float prior_weight, void* cuda_stream, r3_tpe_t** out)
{
    if (out) *out = nullptr;
    if (!X || !y || !levels || !out) {
        set_error("r3_tpe_fit: NULL argument");
        return R3_ERR_INVALID_ARG;
    }
    if (n < 1 || n > kTpeMaxN || d < 1 || d > kMaxD) {
        set_error("r3_tpe_fit: need 1 <= n <= %d and 1 <= d <= %d (got n=%d, d=%d)", kTpeMaxN, kMaxD, n, d);
        return R3_ERR_INVALID_ARG;
    }
    if (!(gamma > 0.f && gamma <= 1.f) || !(prior_weight > 0.f) || !isfinite(prior_weight)) {
        set_error("r3_tpe_fit: need 0 < gamma <= 1 and a finite prior_weight > 0");
        return R3_ERR_INVALID_ARG;
    }
    for (int j = 0; j < d; ++j)
        if (levels[j] != 0 && (abs(levels[j]) < 2 || abs(levels[j]) > kTpeMaxLevels)) {
            set_error("r3_tpe_fit: levels[%d] = %d; allowed are 0, 2..%d and -%d..-2", j, levels[j], kTpeMaxLevels,
                      kTpeMaxLevels);
            return R3_ERR_INVALID_ARG;
        }
    r3_tpe* t = new (std::nothrow) r3_tpe;
    if (!t) {
        set_error("r3_tpe_fit: out of host memory");
        return R3_ERR_ALLOC;
    }
    t->n = n;
    t->d = d;
    t->prior_weight = prior_weight;
    const long long ng = (long long)ceil((double)gamma * (double)n);
    t->n_good = (int)(ng < 1 ? 1 : (ng > n ? n : ng));
    t->levels.assign(levels, levels + d);
    const r3_status_t st = tpe_fit_impl(t, X, y, (cudaStream_t)cuda_stream);
    if (st != R3_OK) {
        tpe_destroy(t);
        return st;
    }
    *out = t;
    return R3_OK;
}

r3_status_t r3_tpe_score(r3_tpe_t* tpe, const float* Xcand, long long m, float* score, void* cuda_stream)
{
    if (!tpe || !Xcand || !score) {
        set_error("r3_tpe_score: NULL argument");
        return R3_ERR_INVALID_ARG;
    }
    if (m < 1 || m >= (1ll << 31)) {
        set_error("r3_tpe_score: need 1 <= m < 2^31 (got %lld)", m);
        return R3_ERR_INVALID_ARG;
    }
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const bool all_tables = tpe->tabled == tpe->d;
    if (all_tables && (tpe->d % 4 != 0 || reinterpret_cast<uintptr_t>(Xcand) % 16 != 0)) {
        // two candidates per thread when that still gives every SM several blocks
        const long long tiles2 = (m + 2ll * kScoreThreads - 1) / (2ll * kScoreThreads);
        const long long tiles1 = (m + kScoreThreads - 1) / kScoreThreads;
        if (tiles2 >= 148ll * 8)
            R3_LAUNCH(tpe_lookup_score_kernel<2>, (unsigned)std::min<long long>(tiles2, 148ll * 16), kScoreThreads, 0, stream,
                      Xcand, m, tpe->d, tpe->levels_d, tpe->table_d, score, tpe->status_d);
        else
            R3_LAUNCH(tpe_lookup_score_kernel<1>, (unsigned)tiles1, kScoreThreads, 0, stream, Xcand, m, tpe->d, tpe->levels_d,
                      tpe->table_d, score, tpe->status_d);
        return R3_OK;
    }
    if (all_tables) {
        // every dimension is a look-up: stream the pool with whole-row loads
        const int d4 = tpe->d / 4;
#define R3_TPE_TABLE(LPC)                                                                                      \
    do {                                                                                                       \
        const int iters = (d4 + LPC - 1) / LPC;                                                                \
        const size_t smem = sizeof(float) * (size_t)iters * 4 * 32 * (kTpeMaxLevels + 1);                      \
        if (smem > 48 * 1024)                                                                                  \
            R3_CUDA_TRY(cudaFuncSetAttribute(tpe_table_score_kernel<LPC>,                                      \
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));         \
        const unsigned grid = 148 * (smem > 56 * 1024 ? 2 : 4);                                                \
        R3_LAUNCH(tpe_table_score_kernel<LPC>, grid, 256, smem, stream, Xcand, m, tpe->d, tpe->levels_d,       \
                  tpe->table_d, score, tpe->status_d);                                                         \
    } while (0)
        if (d4 >= 32) R3_TPE_TABLE(32);
        else if (d4 >= 16) R3_TPE_TABLE(16);
        else if (d4 >= 8) R3_TPE_TABLE(8);
        else if (d4 >= 4) R3_TPE_TABLE(4);
        else if (d4 >= 2) R3_TPE_TABLE(2);
        else R3_TPE_TABLE(1);
#undef R3_TPE_TABLE
        return R3_OK;
    }
    if (tpe->resident) {
        // the whole model in shared memory.  Sixteen blocks per SM's worth of grid (several waves of short
        // blocks) measured up to 8 % faster than one resident wave walking the tiles: the model is a small
        // read from L2 and the finer grain balances the SMs better.
        const long long tiles2 = (m + 2ll * kScoreThreads - 1) / (2ll * kScoreThreads);
        const long long tiles1 = (m + kScoreThreads - 1) / kScoreThreads;
#define R3_TPE_RESIDENT(R, SPLIT, TILES)                                                                       \
    do {                                                                                                       \
        const size_t smem = sizeof(float) * 3 * resident_padded(tpe->total, tpe->d) +                          \
                            sizeof(int4) * (tpe->d - (SPLIT ? tpe->tabled : 0)) +                              \
                            sizeof(int) * (2 * (size_t)tpe->d + 1);                                            \
        if (smem + sizeof(Features) > 48 * 1024)   /* static and dynamic together */                           \
            R3_CUDA_TRY(cudaFuncSetAttribute(tpe_score_resident_kernel<R, SPLIT>,                              \
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));         \
        const unsigned grid = (unsigned)std::min<long long>(TILES, 148ll * 16);                                \
        R3_LAUNCH((tpe_score_resident_kernel<R, SPLIT>), grid, kScoreThreads, smem, stream, Xcand, m, tpe->d,  \
                  tpe->levels_d, tpe->tabled, tpe->offs_d, tpe->packed_d, tpe->total, tpe->table_d, score,     \
                  tpe->status_d);                                                                              \
    } while (0)
        // two candidates per thread when that still gives every SM several blocks; which loop: see the kernel
        if (tiles2 < 148ll * 8)
            R3_TPE_RESIDENT(1, true, tiles1);
        else if (tpe->tabled >= 6 * (tpe->d - tpe->tabled))
            R3_TPE_RESIDENT(2, true, tiles2);
        else
            R3_TPE_RESIDENT(2, false, tiles2);
#undef R3_TPE_RESIDENT
        return R3_OK;
    }
    // Two candidates per thread (one shared-memory read serves both) when that still gives every SM
    // several blocks; one per thread for small pools.  More per thread measured slower on the full pool
    // (fewer, longer blocks balance worse over the 148 SMs).
    const long long tiles2 = (m + 2ll * kScoreThreads - 1) / (2ll * kScoreThreads);
    if (tiles2 >= 148ll * 4) {
        const unsigned grid = (unsigned)(tiles2 < 148ll * 64 ? tiles2 : 148ll * 64);
        R3_LAUNCH(tpe_score_kernel<2>, grid, kScoreThreads, 0, stream, Xcand, m, tpe->n, tpe->d, tpe->n_good,
                  tpe->levels_d, tpe->tabled, tpe->comps_d, tpe->counts_d, tpe->table_d, score, tpe->status_d);
    } else {
        const long long tiles1 = (m + kScoreThreads - 1) / kScoreThreads;
        R3_LAUNCH(tpe_score_kernel<1>, (unsigned)tiles1, kScoreThreads, 0, stream, Xcand, m, tpe->n, tpe->d,
                  tpe->n_good, tpe->levels_d, tpe->tabled, tpe->comps_d, tpe->counts_d, tpe->table_d, score, tpe->status_d);
    }
    return R3_OK;
}

r3_status_t r3_tpe_check(r3_tpe_t* tpe, void* cuda_stream)
{
    if (!tpe) {
        set_error("r3_tpe_check: NULL handle");
        return R3_ERR_INVALID_ARG;
    }
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    R3_CUDA_TRY(cudaMemcpyAsync(tpe->status_h, tpe->status_d, sizeof(int), cudaMemcpyDeviceToHost, stream));
    R3_CUDA_TRY(cudaMemsetAsync(tpe->status_d, 0, sizeof(int), stream));
    R3_CUDA_TRY(cudaStreamSynchronize(stream));
    if (*tpe->status_h & DEV_NONFINITE) {
        set_error("r3_tpe_score: a candidate contains NaN or Inf");
        return R3_ERR_NONFINITE;
    }
    return R3_OK;
}

r3_status_t r3_tpe_get_model(r3_tpe_t* tpe, int* n_good, int* order, float* comps, int* counts, float* table)
{
    if (!tpe) {
        set_error("r3_tpe_get_model: NULL handle");
        return R3_ERR_INVALID_ARG;
    }
    R3_CUDA_TRY(cudaDeviceSynchronize());
    if (n_good) *n_good = tpe->n_good;
    if (order) R3_CUDA_TRY(cudaMemcpy(order, tpe->order_d, sizeof(int) * tpe->n, cudaMemcpyDeviceToHost));
    if (comps)
        R3_CUDA_TRY(cudaMemcpy(comps, tpe->comps_d, sizeof(float4) * (size_t)tpe->d * (tpe->n + 2),
                               cudaMemcpyDeviceToHost));
    if (counts) R3_CUDA_TRY(cudaMemcpy(counts, tpe->counts_d, sizeof(int) * 2 * (size_t)tpe->d, cudaMemcpyDeviceToHost));
    if (table)
        R3_CUDA_TRY(cudaMemcpy(table, tpe->table_d, sizeof(float) * (size_t)tpe->d * kTpeMaxLevels,
                               cudaMemcpyDeviceToHost));
    return R3_OK;
}

void r3_tpe_free(r3_tpe_t* tpe) { tpe_destroy(tpe); }

}  // extern "C"
