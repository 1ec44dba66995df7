// What a fit derives from the inverse factor, in one cooperatively launched kernel:
//   alpha = W^T (W y)                     FP64 and FP32
//   |W|_2, times 1.5                      twelve power iterations on W^T W (the engines' error estimates)
//   W rounded to FP32, max |W|            for the scoring engines' operands
// A GP is served by a team of blocks that meet at a barrier of their own.  A pass u = W v, v' = W^T u reads W twice: rows
// by warps (dealt to and fro, so that every warp gets the same length), then columns by blocks, 16 at a time.
// The weights ride on the first pass.  Vectors sit in shared memory; the norm of a new vector divides the next product, so
// that normalising costs no barrier.
//
// Bound: W from L2, 26 times 4 n^2 bytes, and 25 barriers.  Up to 544 observations a cluster of blocks per GP keeps W in
// shared memory instead and exchanges one vector per pass (one GP of 64 observations: 22 us, 29 us by one block; of 100 to
// 180: 26 us, 53 us by one block; of 300 with the launch: 44 us, 93 us by a team).  Before, 57 launches of three kernels per
// pass: 0.90 ms for one GP of 4096 observations (now 0.31 ms), 0.12 ms and 0.2 ms of launches for one of 64.
#include <cooperative_groups.h>

#include <algorithm>

#include "r3_f64.cuh"
#include "r3_internal.cuh"
#include "r3_tc_common.cuh"

namespace r3 {

namespace {

namespace cg = cooperative_groups;

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
    WaitRule wait;
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
                const double2 w = __ldcg(reinterpret_cast<const double2*>(Wr + R3_IDX(k, npad - 1, a.status)));
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
                *reinterpret_cast<float2*>(o + R3_IDX(k, npad - 1, a.status)) = f;
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
        const double2 x = __ldcg(reinterpret_cast<const double2*>(Wg + (size_t)R3_IDX(i, npad, a.status) * npad));
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

// One cluster of R blocks per GP, W in their shared memory: row i in block i mod R, packed to the diagonal.  A block forms
// its own rows' products u_i = W_i . x and at once their share sum u_i W_i of the new vector.  The shares are written
// straight into all blocks' shared memory (asynchronous stores that count on the receiver's mbarrier), which is the only
// exchange of a pass, and every block adds them up in the same order.  Two sets of shares: a block sends the next set only
// after it has read this one, so whoever sends the one after next has seen that.
// Eight lanes take a row (128 contiguous bytes), a thread two columns and every P-th of the block's rows.
// Bound: instructions issued by all warps alike, so a short history gets few warps and everything that depends only on the
// thread is worked out before the passes.
constexpr int kClusterThreads = 512;   // at most
constexpr int kMaxParts = 4;
__host__ __device__ inline int cluster_threads(int npad) { return npad <= 128 ? 128 : npad <= 256 ? 256 : 512; }
__host__ __device__ inline int cluster_parts(int npad) { return min(kMaxParts, cluster_threads(npad) / (npad / 2)); }
__host__ __device__ inline int packed_doubles(int npad, int R) { return npad / 2 * (npad / R + 1); }
constexpr size_t kClusterSmem = 226 * 1024;   // dynamic; a block's static arrays take a little more
inline size_t cluster_smem(int npad, int R)   // W, x, the shares, the parts of a share, u
{
    return sizeof(double) * ((size_t)packed_doubles(npad, R) + npad + 2 * R * npad + cluster_parts(npad) * npad + npad / R);
}

__device__ __forceinline__ uint32_t in_block(uint32_t addr, int block)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(block));
    return r;
}
__device__ __forceinline__ void send(uint32_t dst, uint32_t bar, double2 v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
                 "l"(__double_as_longlong(v.x)), "l"(__double_as_longlong(v.y)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool arrived(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}

__device__ __forceinline__ void count_as_arrived(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

template <int R>
__global__ void __launch_bounds__(kClusterThreads, 1) weights_cluster_kernel(const WeightArgs a)
{
    extern __shared__ __align__(16) double vec[];
    __shared__ double warp_sums[kClusterThreads / 32];
    __shared__ int warp_tops[kClusterThreads / 32];
    __shared__ __align__(8) unsigned long long bars[2];
    __shared__ int gave_up;   // a wait ran out in some block of the cluster
    __shared__ int sent;      // passes whose shares this block has sent
    cg::cluster_group cluster = cg::this_cluster();
    const int r = (int)cluster.block_rank(), g = blockIdx.x / R, threads = blockDim.x, warps = threads / 32;
    const int t = threadIdx.x, lane = t % 32, warp = t / 32, npad = a.npad, n = a.n, rows = npad / R, half = npad / 2;
    const int P = cluster_parts(npad), even = (r & ~1) + 2;
    const int packed = packed_doubles(npad, R);
    double *Ws = vec, *x = Ws + packed, *shares = x + npad, *parts = shares + 2 * R * npad, *u = parts + P * npad;
    auto at = [&](int q) { return R / 2 * q * (q - 1) + q * even; };   // start of row R q + r: its length is even
    const double* Wg = a.W + (size_t)g * npad * npad;
    for (int q = warp; q < rows; q += warps)
        for (int c = lane; c <= (R * q + r) / 2; c += 32)
            cp_async16(Ws + R3_IDX(at(q) + 2 * c, packed - 1, a.status),
                       Wg + (size_t)R3_IDX(R * q + r, npad, a.status) * npad + R3_IDX(2 * c, npad - 1, a.status));
    cp_async_commit();
    for (int j = t; j < npad; j += threads) x[j] = j < n ? (double)a.y[(size_t)g * n + j] : 0.0;
    if (t == 0) {
        mbar_init(smem_u32(&bars[0]), 1);
        mbar_init(smem_u32(&bars[1]), 1);
        gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (t < kClusterThreads / 32) {
        warp_sums[t] = 0.0;
        warp_tops[t] = 0;
    }
    cp_async_wait<0>();
    cluster.sync();
    if (a.W32 || a.wmax) {
        float top = 0.f;
        for (int q = warp; q < rows; q += warps) {
            const int i = R * q + r;
            for (int c = lane; c < half; c += 32) {
                float2 f = make_float2(0.f, 0.f);
                if (c <= i / 2) {
                    const double2 w = *reinterpret_cast<const double2*>(Ws + R3_IDX(at(q) + 2 * c, packed - 1, a.status));
                    f = make_float2((float)w.x, (float)w.y);
                }
                if (i < n) top = fmaxf(top, fmaxf(fabsf(f.x), fabsf(f.y)));
                if (a.W32) *reinterpret_cast<float2*>(a.W32 + ((size_t)g * npad + i) * npad + 2 * c) = f;
            }
        }
        if (a.wmax) {
            const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
            if (lane == 0 && m) atomicMax(&a.wmax[g], m);
        }
    }
    // the sum of all threads' values, to every thread
    auto total = [&](double v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) warp_sums[warp] = v;
        __syncthreads();
        double all = 0.0;
        for (int w = 0; w < warps; ++w) all += warp_sums[w];
        return all;
    };
    // this thread's columns 2 c and 2 c + 1, its first row there and the distance to the next ones in W
    const int c = t % half, p = t / half, lots = threads / half;
    const int q0 = p < P ? max(0, (2 * c - r + R - 1) / R) + p : rows;
    const int off0 = at(q0) + 2 * c, step0 = at(q0 + P) - at(q0), grow = R * P * P;
    const bool second = rows > threads / 8;
    const uint32_t mine = smem_u32(shares + r * npad + 2 * c);
    double2 v = make_double2(0.0, 0.0);   // (thread < half) the new vector's columns 2 t and 2 t + 1
    bool late = false;                    // a bounded wait ran out, here or in another block of the cluster
    const int sends = a.wait.withhold && r == R - 1 ? 1 : a.iters + 1;   // (a test keeps the last block's shares back)
    auto pass = [&](double scale, int turn) {   // x, v <- W^T (scale W x)
        for (int q = t / 8; q < rows; q += threads / 8) {
            const int i = R * q + r, m = i < n ? i / 2 : -1;
            const double* w = Ws + at(q);
            double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
            for (int k = t % 8; k <= m; k += 8) {
                const double2 e = *reinterpret_cast<const double2*>(w + R3_IDX(2 * k, packed - 1 - at(q), a.status)),
                              f = *reinterpret_cast<const double2*>(x + R3_IDX(2 * k, npad - 1, a.status));
                s0 = fma(e.x, f.x, s0);
                s1 = fma(e.y, f.y, s1);
            }
            s0 += s1;
            const unsigned mask = 0xffu << (lane & 24);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s0 += __shfl_xor_sync(mask, s0, o);
            if (t % 8 == 0) u[q] = s0 * scale;
            if (!second) break;
        }
        __syncthreads();
        const int buffer = turn & 1;
        const uint32_t bar = smem_u32(&bars[buffer]);
        if (t == 0) mbar_arrive_expect_tx(bar, (uint32_t)(R * npad * sizeof(double)));
        if (p < P) {
            double2 s = make_double2(0.0, 0.0);
            int off = off0, step = step0;
#pragma unroll 4
            for (int q = q0; q < rows; q += P) {   // the rows from the diagonal on
                const double2 e = *reinterpret_cast<const double2*>(Ws + R3_IDX(off, packed - 1, a.status));
                const double uq = u[R3_IDX(q, rows, a.status)];
                s.x = fma(e.x, uq, s.x);
                s.y = fma(e.y, uq, s.y);
                off += step;
                step += grow;
            }
            *reinterpret_cast<double2*>(parts + p * npad + 2 * c) = s;
        }
        __syncthreads();
        if (p < min(lots, R) && turn < sends) {   // two columns to every lots-th block
            double2 s = *reinterpret_cast<const double2*>(parts + 2 * c);
#pragma unroll
            for (int k = 1; k < kMaxParts; ++k)
                if (k < P) {
                    const double2 e = *reinterpret_cast<const double2*>(parts + k * npad + 2 * c);
                    s.x += e.x;
                    s.y += e.y;
                }
            const uint32_t dst = mine + buffer * (uint32_t)(R * npad * sizeof(double));
#pragma unroll 1
            for (int b = p; b < R; b += lots) send(in_block(dst, b), in_block(bar, b), s);
        }
        if (t < half) {
            const uint32_t parity = (turn >> 1) & 1;
            if (!arrived(bar, parity)) {
                const long long t0 = clock64();
                while (!arrived(bar, parity)) {
                    late = *reinterpret_cast<volatile int*>(&gave_up) != 0;
                    if (!late && clock64() - t0 > a.wait.cycles) {
                        late = true;
                        atomicOr(a.status, DEV_TIMEOUT);
                        for (int b = 0; b < R; ++b) *reinterpret_cast<volatile int*>(cluster.map_shared_rank(&gave_up, b)) = 1;
                    }
                    if (late) break;
                }
            }
            const double* from = shares + buffer * R * npad + 2 * t;
            v = make_double2(0.0, 0.0);
#pragma unroll
            for (int b = 0; b < R; ++b) {
                const double2 e = *reinterpret_cast<const double2*>(from + b * npad);
                v.x += e.x;
                v.y += e.y;
            }
            *reinterpret_cast<double2*>(x + 2 * t) = v;
        }
    };
    double sum = 0.0, before = 0.0, scale = 1.0;
    int entered = 0;   // passes begun
#pragma unroll 1
    for (int turn = 0; turn <= a.iters; ++turn) {
        pass(scale, turn);
        entered = turn + 1;
        if (turn == 0) {
            if (t < half) {
                if (r == 0) {
                    *reinterpret_cast<double2*>(a.alpha64 + (size_t)g * npad + 2 * t) = v;
                    *reinterpret_cast<float2*>(a.alpha32 + (size_t)g * npad + 2 * t) = make_float2((float)v.x, (float)v.y);
                }
                auto start = [&](int j) { return j < n ? 1.0 + 0.37 * ((j * 2654435761u >> 16) & 0xff) / 255.0 : 0.0; };
                v = make_double2(start(2 * t), start(2 * t + 1));
                *reinterpret_cast<double2*>(x + 2 * t) = v;
            }
            if (a.iters == 0) break;
        }
        // 2^-e for the largest exponent e in x: a factor that keeps the iteration in range, without rounding and in a
        // fraction of the time of a norm, its root and the division
        const int top = __reduce_max_sync(0xffffffffu, max(__double2hiint(fabs(v.x)), __double2hiint(fabs(v.y))));
        if (lane == 0) warp_tops[warp] = top;
        if (turn + 1 >= a.iters) {
            before = sum;
            sum = total(fma(v.x, v.x, v.y * v.y));
        }
        if (__syncthreads_or(late)) break;
        if (turn < a.iters) {
            const int e = __reduce_max_sync(0xffffffffu, warp_tops[lane % (kClusterThreads / 32)]) >> 20;
            scale = e == 0 ? 1.0 : __hiloint2double(max(2046 - e, 0) << 20, 0);
        }
    }
    // the growth of the last pass estimates |W|_2^2 from below; 1.5 covers slow convergence
    if (a.iters > 0 && r == 0 && t == 0) a.wnorm[g] = before > 0.0 ? 1.5 * sqrt(sqrt(sum) / (sqrt(before) * scale)) : 0.0;
    // No block leaves while another's shares may still be on their way to it.  A block that has waited for all its passes has
    // them all; after this barrier everyone else's have been sent as well.
    if (t == 0) sent = min(entered, sends);
    cluster.sync();
    if (gave_up) {   // said in every block before the barrier, so all see the same
        // All blocks have sent the shares of the passes before the last one begun here.  Of that pass, and of the one after
        // it (begun by blocks that got their shares), those that were sent are waited for.
        if (t == 0) {
            int missing = 0, ahead = 0;
            for (int b = 0; b < R; ++b) {
                const int theirs = *cluster.map_shared_rank(&sent, b);
                missing += theirs < entered ? 1 : 0;
                ahead += theirs > entered ? 1 : 0;
            }
            const uint32_t share = (uint32_t)(npad * sizeof(double));
            auto land = [&](int turn) {
                const long long t0 = clock64();
                while (!arrived(smem_u32(&bars[turn & 1]), (turn >> 1) & 1) && clock64() - t0 < 2000000) {}
            };
            if (missing) count_as_arrived(smem_u32(&bars[(entered - 1) & 1]), missing * share);
            land(entered - 1);
            if (ahead) {
                mbar_arrive_expect_tx(smem_u32(&bars[entered & 1]), ahead * share);
                land(entered);
            }
        }
        cluster.sync();
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
            return team_barrier(a.barrier + g, target, (unsigned)a.team, a.status, a.wait);
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
    a.wait = p.wait;
    int sms = 148;
    R3_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    // W in shared memory, as far as that goes (R = 2: 320 observations, R = 8: 544).  Eight blocks per GP while that leaves
    // at most two on a multiprocessor, or where two do not hold W: one GP of 300 44 us (R = 2: 86, teams: 93), 64 of 300
    // 201 us (R = 2: 88, teams: 238), 64 of 512 348 us (teams: 479).  Weights alone take one pass, for which loading W
    // pays less: with more than 320 observations the team has them sooner if every GP gets a full one (8 of 512: 15 us, R = 8: 18).
    const int resident2 = 2 * sms, R = 8 * p.batch <= resident2 || cluster_smem(p.npad, 2) > kClusterSmem ? 8 : 2;
    const bool full_teams = p.batch * (p.npad / kCols) <= resident2;
    if (cluster_smem(p.npad, R) <= kClusterSmem && (a.iters > 0 || p.npad <= 320 || !full_teams)) {
        auto kernel = R == 8 ? weights_cluster_kernel<8> : weights_cluster_kernel<2>;
        R3_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmem));
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = R;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(R * p.batch);
        cfg.blockDim = dim3(cluster_threads(p.npad));
        cfg.dynamicSmemBytes = cluster_smem(p.npad, R);
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        R3_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, a));
        ++g_launches;
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
