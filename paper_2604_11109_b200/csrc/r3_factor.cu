// Covariance matrix, Cholesky factor and inverse factor of every GP of a handle, in one cooperatively launched kernel:
//   K = k(X,X) + noise*I   by direct differences, computed where it is consumed and never stored
//   K = L L^T,  W = L^-1
// in FP64, for a whole history (r3_gp_fit) or for the rows that an append adds (the rows of L and W above them are
// taken as given, so that an append is the tail of the same computation, not another algorithm).
//
// The matrices are cut into 64 x 64 tiles and the work into tasks, one tile of L or W each:
//   L(i,j), i > j   A = K(i,j) - sum_{k<j} L(i,k) L(j,k)^T, then A L(j,j)^-T by forward substitution
//   L(j,j)          the same sum, factored in shared memory; W(j,j) = L(j,j)^-1 follows
//   W(i,c), i > c   -W(i,i) sum_{c<=k<i} L(i,k) W(k,c)
// Blocks draw tasks from a ticket counter in the order: for every j the diagonal tile of column j of L, row j - 1 of W,
// the rest of column j.  A task depends only on tasks before it, all blocks are resident, and a block works its tasks off
// one by one, so some block can always go on.  The row of W is work for the blocks while the diagonal tile is factored (64
// GPs of 512: 515 to 473 us, one of 1000 336 to 305 us against row j after column j; with L(j+1,j) and L(j+1,j+1) before
// the rest of column j 2048 observations gain 9 % and 64 GPs of 512 lose 3 %).  Progress is one counter per row of L (its
// tiles finish from left to right) and one per column of W (from top to bottom); a task adds up the products whose
// operands are there and waits for the next.
// A tile of L is handed out in halves of 32 columns: the left half of a column's tiles is solved, stored and multiplied
// while one warp factors the diagonal tile's second panel (300 observations: 118 -> 93 us; 1000: fit 621 -> 552 us).
// So a tile is written once and read as an operand, nothing is updated in place, and the factor's critical path --
// 64 columns in shared memory, one substitution, one product -- runs while the other blocks are busy with tiles far
// from it.  Products run on the FP64 tensor path with three 16-deep operand stages in flight.
//
// (The substitution is deliberate: a product with the explicit inverse of L(j,j) loses the small entries of an
// ill-conditioned factor, and the log-determinant of noise-free smooth data came out wrong in the third digit.)
//
// Bound: FP64 rate for long histories, the chain of diagonal blocks for short ones.  One GP of 4096 observations (64
// features): 2.9 ms, 32 TFLOP/s of FP64 without the exponentials (a sequence of 290 launches with 4x4 register tiles and
// recursive doubling for the inverse: 7.2 ms); 300 observations 0.09 ms (0.41 ms); 64 GPs of 512 0.47 ms (1.26 ms).
// An append of 128 to 3968 (it was triangular products, a Schur complement and their corrections): 0.6 ms (2.0 ms).
#include <algorithm>

#include "r3_f64.cuh"
#include "r3_internal.cuh"

namespace r3 {

namespace {

constexpr int TB = kFactorTile;
constexpr int kThreads = 256;   // eight warps, 16 x 32 results each
constexpr int kStages = 3;
constexpr int kLd = 68;         // leading dimension of whole tiles in shared memory: 4 mod 16, like the stages'
constexpr size_t kFactorSmem = sizeof(double) * 2 * TB * kLd;   // two tiles; the stages take less
constexpr int kMaxTiles = kMaxN / TB;

struct FactorArgs {
    const float *X, *ell, *sf2, *sn2;
    int batch, n, d, npad, T, i0;   // T tile rows; those below i0 are finished
    double *L, *W;                  // [batch][npad][npad]
    int *lprog;                     // [batch][T] finished half tiles (32 columns) of each row of L
    int *wprog;                     // [batch][T] one past the last finished half tile of each column of W
    unsigned* ticket;
    int* status;
    WaitRule wait;
    int first[kMaxTiles + 2];       // tasks per GP before step j
};

__device__ __forceinline__ int load_acquire_int(const int* p) { return (int)load_acquire(reinterpret_cast<const unsigned*>(p)); }
__device__ __forceinline__ void store_release_int(int* p, int v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Waits (one thread) until *p >= want and returns what it saw; -1 when the wait ran out.  Blocks whose operands never come
// begin to wait within the time of the tasks that still can be done, so a failed factorisation costs that and one limit.
__device__ __forceinline__ int wait_progress(const int* p, int want, int* status, const WaitRule& rule)
{
    int v = load_acquire_int(p);
    if (v >= want) return v;
    const long long t0 = clock64();
    while (true) {
        __nanosleep(40);
        v = load_acquire_int(p);
        if (v >= want) return v;
        if (clock64() - t0 > rule.cycles) {
            atomicOr(status, DEV_TIMEOUT);
            return -1;
        }
    }
}

struct Shared {
    int task, ready, ok;
    double rinv[TB];   // reciprocal roots of the diagonal block's pivots
};

// This thread's accumulators, -K(i,j): rows wm + 8 a + l / 4, columns wn + 8 b + 2 (l % 4) + h.
__device__ __forceinline__ void gram_tile(const FactorArgs& a, int g, int ti, int tj, unsigned char* smem, double (&c)[2][4][2])
{
    double* xi = reinterpret_cast<double*>(smem);   // [64][33]
    double* xj = xi + TB * 33;
    double* il = xj + TB * 33;                      // [32]
    const int t = threadIdx.x, w = t / 32, l = t % 32;
    const int wm = (w % 4) * 16, wn = (w / 4) * 32;
    const int n = a.n, d = a.d;
    const float* Xg = a.X + (size_t)g * n * d;
    double r2[2][4][2] = {};
    for (int c0 = 0; c0 < d; c0 += 32) {
        __syncthreads();
        // all of a thread's loads are under way before the first is stored
        const int f0 = t % 32, q0 = t / 32;
        float vi[8], vj[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int gi = ti * TB + q0 + 8 * e, gj = tj * TB + q0 + 8 * e;
            vi[e] = (gi < n && c0 + f0 < d) ? __ldg(Xg + R3_IDX((size_t)gi * d + c0 + f0, (size_t)n * d, a.status)) : 0.f;
            vj[e] = (gj < n && c0 + f0 < d) ? __ldg(Xg + R3_IDX((size_t)gj * d + c0 + f0, (size_t)n * d, a.status)) : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            xi[(q0 + 8 * e) * 33 + f0] = (double)vi[e];
            xj[(q0 + 8 * e) * 33 + f0] = (double)vj[e];
        }
        // FP64 reciprocal of the lengthscale: one rounding more than a division per difference, a third of its time
        if (t < 32) il[t] = (c0 + t < d) ? 1.0 / (double)a.ell[(size_t)g * d + c0 + t] : 0.0;
        __syncthreads();
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
    const double sf2 = (double)a.sf2[g], sn2 = (double)a.sn2[g];
    int twin = a.n;   // a row that repeats an earlier one
#pragma unroll 1
    for (int j = 0; j < 4; ++j)   // not unrolled: four square roots and exponentials at a time are enough to overlap
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = ti * TB + wm + 8 * i + l / 4, col = tj * TB + wn + 8 * j + 2 * (l % 4) + h;
                double r = 0.0;
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) r = jj == j ? r2[i][jj][h] : r;
                const double s = sqrt(5.0) * sqrt(r);
                double v = sf2 * fma(s, fma(s, 1.0 / 3.0, 1.0), 1.0) * exp(-s);
                if (row == col) v += sn2;
                else if (r == 0.0 && col < row) twin = min(twin, row);
                if (row >= n || col >= n) v = row == col ? 1.0 : 0.0;   // the identity beyond the history
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) c[i][jj][h] = jj == j ? -v : c[i][jj][h];
            }
    // Two equal rows whose noise is lost in the diagonal's rounding: K is singular whatever sign its pivots come out with
    if (twin < n && sf2 + sn2 == sf2) {
        atomicOr(&a.status[0], DEV_NOT_PD);
        atomicMin(&a.status[1], twin);
    }
}

// One 16-deep step: A fragments at pa (row stride lda), B fragments either [column][k] (NT) or [k][column].
template <bool NT>
__device__ __forceinline__ void mma_step(const double* pa, int lda, const double* pb, int ldb, double (&c)[2][4][2])
{
#pragma unroll
    for (int kk = 0; kk < 16; kk += 4) {
        double fa[2], fb[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) fa[i] = pa[i * 8 * lda + kk];
#pragma unroll
        for (int j = 0; j < 4; ++j) fb[j] = NT ? pb[j * 8 * ldb + kk] : pb[kk * ldb + j * 8];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) dmma(c[i][j], fa[i], fb[j]);
    }
}

// c += sum over tile columns [k0, k1) of L(i,k) B(k), with B(k) = L(j,k)^T (NT) or W(k,j).  Waits for the operands as it
// goes.  Returns false when a wait ran out.
template <bool NT>
__device__ __forceinline__ bool accumulate(const FactorArgs& a, int g, int i, int j, int k0, int k1, unsigned char* smem,
                                           Shared& sh, double (&c)[2][4][2])
{
    constexpr int kLdb = NT ? kStageLd : kLd;             // B stage: [64][20] or [16][68]
    constexpr int kBStage = NT ? TB * kStageLd : 16 * kLd;
    double* sA = reinterpret_cast<double*>(smem);
    double* sB = sA + kStages * TB * kStageLd;
    const int t = threadIdx.x, w = t / 32, l = t % 32;
    const int wm = (w % 4) * 16, wn = (w / 4) * 32, npad = a.npad;
    const double* Lg = a.L + (size_t)g * npad * npad;
    const double* Wg = a.W + (size_t)g * npad * npad;
    const int* li = a.lprog + (size_t)g * a.T + i;
    const int* lj = a.lprog + (size_t)g * a.T + j;
    const int* wj = a.wprog + (size_t)g * a.T + j;
    // thread 0: the number of half tiles whose operands are there (at least `want`), -1 if a wait ran out
    auto poll = [&](int want) {
        int v = i < a.i0 ? 2 * a.T : wait_progress(li, want, a.status, a.wait);
        if (v < 0) return -1;
        int u;
        if (NT) u = j < a.i0 ? 2 * a.T : (j == i ? v : wait_progress(lj, want, a.status, a.wait));
        else u = want <= 2 * a.i0 ? 2 * a.i0 : wait_progress(wj, want, a.status, a.wait);
        return u < 0 ? -1 : min(u, v);
    };
    auto load = [&](int s, int k) {   // stage s <- columns k .. k + 15
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            const int e = t + kThreads * it, r = e / 8, q = e % 8;
            const bool oki = i * TB + r < npad, okj = j * TB + r < npad;
            auto at = [&](int row, int col) { return (size_t)R3_IDX(row, npad, a.status) * npad + R3_IDX(col, npad - 1, a.status); };
            cp_async16(sA + (s * TB + r) * kStageLd + 2 * q, Lg + at(oki ? i * TB + r : 0, k + 2 * q), oki);
            if (NT) {
                cp_async16(sB + s * kBStage + r * kLdb + 2 * q, Lg + at(okj ? j * TB + r : 0, k + 2 * q), okj);
            } else {
                const int rr = e / 32, qq = e % 32;
                cp_async16(sB + s * kBStage + rr * kLdb + 2 * qq, Wg + at(k + rr, j * TB + 2 * qq));
            }
        }
    };
    const int s0 = k0 * 4, s1 = k1 * 4;   // 16-deep steps
    if (s0 >= s1) return true;
    __syncthreads();                      // the stages' bytes were last used for something else
    if (t == 0) sh.ready = poll(2 * k0 + 1);
    __syncthreads();
    int ready = sh.ready;
    if (ready < 0) return false;
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
        load(s, (s0 + s) * 16);           // the first half tile has two steps
        cp_async_commit();
    }
    for (int s = s0; s < s1; ++s) {
        const int nx = s + kStages - 1;   // the step to fetch now
        cp_async_wait<kStages - 2>();
        const bool ask = nx < s1 && nx / 2 >= ready;
        if (ask && t == 0) sh.ready = poll(nx / 2 + 1);
        __syncthreads();
        if (ask) {
            ready = sh.ready;
            if (ready < 0) {
                cp_async_wait<0>();
                return false;
            }
        }
        if (nx < s1) load((nx - s0) % kStages, nx * 16);
        cp_async_commit();
        const int st = (s - s0) % kStages;
        mma_step<NT>(sA + (st * TB + wm + l / 4) * kStageLd + l % 4, kStageLd,
                     NT ? sB + st * kBStage + (wn + l / 4) * kLdb + l % 4 : sB + st * kBStage + (l % 4) * kLdb + wn + l / 4, kLdb, c);
    }
    cp_async_wait<0>();
    __syncthreads();
    return true;
}

// Tile (ti, tj) of a matrix into shared memory (zeros beyond npad), asynchronously.
__device__ __forceinline__ void fetch_tile(const double* Mg, int npad, int ti, int tj, double* dst, int* status)
{
    for (int e = threadIdx.x; e < TB * (TB / 2); e += kThreads) {
        const int r = e / (TB / 2), q = e % (TB / 2);
        const bool ok = ti * TB + r < npad && tj * TB + 2 * q < npad;
        cp_async16(dst + r * kLd + 2 * q, Mg + R3_IDX(ok ? (size_t)(ti * TB + r) * npad + tj * TB + 2 * q : 0, (size_t)npad * npad - 1, status), ok);
    }
    cp_async_commit();
}

__device__ __forceinline__ void store_tile(double* Mg, int npad, int ti, int tj, const double* src, int* status)
{
    for (int e = threadIdx.x; e < TB * (TB / 2); e += kThreads) {
        const int r = e / (TB / 2), q = e % (TB / 2);
        if (ti * TB + r < npad && tj * TB + 2 * q < npad)
            *reinterpret_cast<double2*>(Mg + R3_IDX((size_t)(ti * TB + r) * npad + tj * TB + 2 * q, (size_t)npad * npad - 1, status)) =
                *reinterpret_cast<const double2*>(src + r * kLd + 2 * q);
    }
}

// Of a diagonal tile: columns h .. h + 31 from row h on, as fetch_tile
__device__ __forceinline__ void fetch_half(const double* Mg, int npad, int tj, int h, double* dst, int* status)
{
    for (int e = threadIdx.x; e < (TB - h) * 16; e += kThreads) {
        const int r = h + e / 16, c = h + 2 * (e % 16);
        const bool ok = tj * TB + r < npad && tj * TB + c < npad;
        cp_async16(dst + r * kLd + c, Mg + R3_IDX(ok ? (size_t)(tj * TB + r) * npad + tj * TB + c : 0, (size_t)npad * npad - 1, status), ok);
    }
    cp_async_commit();
}

// Columns h .. h + 31 of a tile, by the threads t of `threads`
__device__ __forceinline__ void store_half(double* Mg, int npad, int ti, int tj, int h, const double* src, int t, int threads,
                                           int* status)
{
    for (int e = t; e < TB * 16; e += threads) {
        const int r = e / 16, c = h + 2 * (e % 16);
        if (ti * TB + r < npad && tj * TB + c < npad)
            *reinterpret_cast<double2*>(Mg + R3_IDX((size_t)(ti * TB + r) * npad + tj * TB + c, (size_t)npad * npad - 1, status)) =
                *reinterpret_cast<const double2*>(src + r * kLd + c);
    }
}

__device__ __forceinline__ void zero_tile(double* Mg, int npad, int ti, int tj, int* status)
{
    for (int e = threadIdx.x; e < TB * (TB / 2); e += kThreads) {
        const int r = e / (TB / 2), q = e % (TB / 2);
        if (ti * TB + r < npad && tj * TB + 2 * q < npad)
            *reinterpret_cast<double2*>(Mg + R3_IDX((size_t)(ti * TB + r) * npad + tj * TB + 2 * q, (size_t)npad * npad - 1, status)) =
                make_double2(0.0, 0.0);
    }
}

__device__ __forceinline__ void park(const double (&c)[2][4][2], double sign, double* dst)
{
    const int w = threadIdx.x / 32, l = threadIdx.x % 32, wm = (w % 4) * 16, wn = (w / 4) * 32;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<double2*>(dst + (wm + 8 * i + l / 4) * kLd + wn + 8 * j + 2 * (l % 4)) =
                make_double2(sign * c[i][j][0], sign * c[i][j][1]);
}

// 1 / sqrt(p) for a normal positive p, NaN otherwise: the hardware's approximation (about 2^-22) and two steps of Newton's
// method for the zero of f(y) = 1/y^2 - p, y <- y - f(y) / f'(y) = y + y (1/2 - p y^2 / 2).  A step takes a relative error e
// to 3/2 e^2, so the second one leaves 2^-84 and its own rounding, at most 2^-52.  Free of branches, so that the rank-one
// update of one column overlaps with the pivot of the next (one GP of 300 observations, fit and 12 evaluations of the
// evidence: 2.42 ms, with CUDA's rsqrt() 2.52 ms).
__device__ __forceinline__ double rsqrt_newton(double p)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(p));
    const double h = -0.5 * p;
    y = fma(y, fma(h * y, y, 0.5), y);
    return fma(y, fma(h * y, y, 0.5), y);
}

__global__ void rsqrt_kernel(const double* __restrict__ p, double* __restrict__ y, long long count)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < count) y[i] = rsqrt_newton(p[i]);
}

// Columns b .. b + 31 of the tile, rows b .. 63 (one warp for 32 rows, two for 64): lane = row, the row's 32 entries in
// registers.  The loop over the columns is not unrolled: the entries move down as they are updated instead, so that the
// step's columns are always the first.  That is twice the multiply-adds (the places beyond the end hold leftovers that
// nothing uses), but straight code for 32 columns is over 20 KB that a block runs once, and fetching it took longer.
// Two columns per step, because the latency of the chain from pivot to pivot is what a diagonal block costs.  With the 2 x 2
// block (p1 . ; s p2) ahead, det = p1 p2 - s^2 and the second pivot is det / p1, so that both reciprocal roots
//     r1 = p1^-1/2,   r2 = (det / p1)^-1/2 = p1 r1 det^-1/2
// are under way together (det is as accurate as the second pivot of column-by-column elimination: its rounding is that of
// p2).  Every lane carries the next block and the entries left of it along, fetched by shuffles a step ahead, so that the
// chain of a step is r2, one column, one update, det and its root, and waits for no broadcast.
// The two panels of a 64 x 64 block: 15,500 cycles; 17,700 column by column, 22,000 with a shuffle in the chain and unrolled
// code.  (Letting the second warp follow by a counter instead of the barrier: 24,000, it falls behind.)
// A pivot's sign decides (gram_tile looks for equal rows without noise, whose pivots are rounding of either sign).
// cols: 16 x 64 doubles of scratch in shared memory.
__device__ __forceinline__ void factor_panel(double* tile, int b, int warps, double* cols, double* rinv, const FactorArgs& a,
                                             int pivot0)
{
    const int w = threadIdx.x / 32, l = threadIdx.x % 32;
    if (w >= warps) return;
    const int row = b + 32 * w + l;
    double x[32];
#pragma unroll
    for (int c = 0; c < 32; c += 2) {
        const double2 v = *reinterpret_cast<const double2*>(tile + row * kLd + b + c);
        x[c] = v.x;
        x[c + 1] = v.y;
    }
    double* out = tile + row * kLd + b;
    auto update = [&](int k, double x0, double x1) {   // the entries move down as they are updated
        const double *c0 = cols + 32 * k, *c1 = c0 + 32;
#pragma unroll
        for (int j = 0; j < 30; j += 2) {
            const double2 u = *reinterpret_cast<const double2*>(c0 + j), v = *reinterpret_cast<const double2*>(c1 + j);
            x[j] = fma(-x1, v.x, fma(-x0, u.x, x[j + 2]));
            x[j + 1] = fma(-x1, v.y, fma(-x0, u.y, x[j + 3]));
        }
    };
    auto meet = [&]() {
        if (warps == 2) asm volatile("bar.sync 1, 64;" ::: "memory");
        else __syncwarp();
    };
    if (w == 0) {
        auto from = [&](double v, int lane) { return __shfl_sync(0xffffffffu, v, lane & 31); };
        double p1 = from(x[0], 0), s = from(x[0], 1), p2 = from(x[1], 1), det = fma(p1, p2, -(s * s));
        double r1 = rsqrt_newton(p1), rd = rsqrt_newton(det);
        // rows k + 2 and k + 3: entries in columns k and k + 1, and their own block, after the updates before column k
        double a0 = from(x[0], 2), a1 = from(x[1], 2), d22 = from(x[2], 2);
        double b0 = from(x[0], 3), b1 = from(x[1], 3), d32 = from(x[2], 3), d33 = from(x[3], 3);
#pragma unroll 1
        for (int k = 0; k < 32; k += 2) {
            const double sq1 = p1 * r1, l21 = s * r1, r2 = sq1 * rd;
            const double la0 = a0 * r1, la1 = fma(-la0, l21, a1) * r2, lb0 = b0 * r1, lb1 = fma(-lb0, l21, b1) * r2;
            const double p1n = fma(-la1, la1, fma(-la0, la0, d22)), sn = fma(-lb1, la1, fma(-lb0, la0, d32)),
                         p2n = fma(-lb1, lb1, fma(-lb0, lb0, d33)), detn = fma(p1n, p2n, -(sn * sn));
            // this lane's entries of the two columns; on the diagonal sqrt(p) from r with one correction step
            // (s = p r, s += r (p - s^2) / 2)
            const double q2 = det * (r1 * r1), sq2 = q2 * r2;
            const double x0 = l == k ? fma(0.5 * r1, fma(-sq1, sq1, p1), sq1) : x[0] * r1;
            const double x1 = l == k + 1 ? fma(0.5 * r2, fma(-sq2, sq2, q2), sq2) : fma(-x0, l21, x[1]) * r2;
            double* c0 = cols + 32 * k;
            if (l > k + 1) {
                c0[l - k - 2] = x0;
                c0[32 + l - k - 2] = x1;
            }
            if (l == k) {
                rinv[b + k] = r1;
                rinv[b + k + 1] = r2;
                c0[31] = l21;
            }
            *reinterpret_cast<double2*>(out + k) = make_double2(l >= k ? x0 : 0.0, l >= k + 1 ? x1 : 0.0);
            meet();
            r1 = rsqrt_newton(p1n);
            rd = rsqrt_newton(detn);
            update(k, x0, x1);
            p1 = p1n;
            s = sn;
            det = detn;
            a0 = from(x[0], k + 4);
            a1 = from(x[1], k + 4);
            d22 = from(x[2], k + 4);
            b0 = from(x[0], k + 5);
            b1 = from(x[1], k + 5);
            d32 = from(x[2], k + 5);
            d33 = from(x[3], k + 5);
        }
        // the pivots' test, once for all: lane = column; beyond the first bad pivot everything is NaN or means nothing
        const double d = tile[row * kLd + row];
        const bool bad = !(d > 0.0) || !isfinite(d);
        const unsigned which = __ballot_sync(0xffffffffu, bad);
        if (which && l == 0) {
            atomicOr(&a.status[0], DEV_NOT_PD);
            atomicMin(&a.status[1], pivot0 + b + __ffs(which) - 1);
        }
    } else {
#pragma unroll 1
        for (int k = 0; k < 32; k += 2) {
            meet();
            const double x0 = x[0] * rinv[b + k], x1 = fma(-x0, cols[32 * k + 31], x[1]) * rinv[b + k + 1];
            *reinterpret_cast<double2*>(out + k) = make_double2(x0, x1);
            update(k, x0, x1);
        }
    }
}

// x L^T = a for 64 rows against the 32 columns at b, two warps, lane = row
__device__ __forceinline__ void solve_panel(double* tile, const double* diag, const double* rinv, int b)
{
    const int row = threadIdx.x;
    if (row >= TB) return;
    double x[32];
#pragma unroll
    for (int c = 0; c < 32; c += 2) {
        const double2 v = *reinterpret_cast<const double2*>(tile + row * kLd + b + c);
        x[c] = v.x;
        x[c + 1] = v.y;
    }
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        x[c] *= rinv[b + c];
#pragma unroll
        for (int k = c + 1; k < 32; ++k) x[k] = fma(-x[c], diag[(b + k) * kLd + b + c], x[k]);
    }
#pragma unroll
    for (int c = 0; c < 32; c += 2) *reinterpret_cast<double2*>(tile + row * kLd + b + c) = make_double2(x[c], x[c + 1]);
}

// tile[:, 32..63] -= tile[:, 0..31] other[32..63, 0..31]^T, rows r0 .. 63
__device__ __forceinline__ void update_right(double* tile, const double* other, int r0)
{
    // warp w: 8 rows (r0 = 0: eight row groups, r0 = 32: four, two warps each taking 16 of the 32 columns)
    const int w = threadIdx.x / 32, l = threadIdx.x % 32;
    const int groups = (TB - r0) / 8, rg = w % groups, half = w / groups, nhalf = 8 / groups;
    const int row = r0 + rg * 8 + l / 4;
    for (int jb = half; jb < 4; jb += nhalf) {
        double c[2] = {0.0, 0.0};
        const double* pa = tile + row * kLd + l % 4;
        const double* pb = other + (32 + jb * 8 + l / 4) * kLd + l % 4;
#pragma unroll
        for (int k = 0; k < 32; k += 4) dmma(c, pa[k], pb[k]);
        double* o = tile + row * kLd + 32 + jb * 8 + 2 * (l % 4);
        o[0] -= c[0];
        o[1] -= c[1];
    }
}

// Inverse of the lower-triangular 32 x 32 block at (b, b): one warp, lane = column
__device__ __forceinline__ void invert_block(const double* diag, const double* rinv, int b, double* out)
{
    const int l = threadIdx.x % 32;
    double x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = i == l ? 1.0 : 0.0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        x[j] *= rinv[b + j];
#pragma unroll
        for (int i = j + 1; i < 32; ++i) x[i] = fma(-diag[(b + i) * kLd + b + j], x[j], x[i]);
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) out[(b + i) * kLd + b + l] = x[i];
}

// out[32..63, 0..31] = -W22 (L21 W11); tmp: 32 x 32 at tmp (leading dimension kLd)
__device__ __forceinline__ void invert_corner(const double* diag, double* out, double* tmp)
{
    const int w = threadIdx.x / 32, l = threadIdx.x % 32, rg = w % 4, half = w / 4;
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        const double* A = pass == 0 ? diag + 32 * kLd : out + 32 * kLd + 32;   // L21, then W22
        const double* B = pass == 0 ? out : tmp;                              // W11, then L21 W11
        for (int jb = half; jb < 4; jb += 2) {
            double c[2] = {0.0, 0.0};
#pragma unroll
            for (int k = 0; k < 32; k += 4)
                dmma(c, A[(rg * 8 + l / 4) * kLd + k + l % 4], B[(k + l % 4) * kLd + jb * 8 + l / 4]);
            double* o = (pass == 0 ? tmp : out + 32 * kLd) + (rg * 8 + l / 4) * kLd + jb * 8 + 2 * (l % 4);
            o[0] = pass == 0 ? c[0] : -c[0];
            o[1] = pass == 0 ? c[1] : -c[1];
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kThreads, 2) factor_kernel(const __grid_constant__ FactorArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Shared sh;
    double* tile0 = reinterpret_cast<double*>(smem);
    double* tile1 = tile0 + TB * kLd;
    const int t = threadIdx.x, w = t / 32, l = t % 32, wm = (w % 4) * 16, wn = (w / 4) * 32;
    const int npad = a.npad, T = a.T;
    const int total = a.first[T + 1] * a.batch;
    auto publish = [&](int* p, int v, bool announce = true) {   // the tile has been stored by all threads
        __syncthreads();
        if (t == 0 && announce) store_release_int(p, v);   // (a release covers what the barrier has made this thread see)
    };
    auto await = [&](const int* p, int want) {
        if (t == 0) sh.ok = wait_progress(p, want, a.status, a.wait);
        __syncthreads();
        return sh.ok >= 0;
    };
    while (true) {
        __syncthreads();
        if (t == 0) sh.task = (int)atomicAdd(a.ticket, 1u);
        __syncthreads();
        const int task = sh.task;
        if (task >= total) return;
        const bool announce = !(a.wait.withhold && task == 0);   // (a test keeps the first tile back)
        int lo = 0, hi = T;   // the step: last j with first[j] * batch <= task
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (a.first[mid] * a.batch <= task) lo = mid;
            else hi = mid - 1;
        }
        // step j: the diagonal tiles of column j, row j - 1 of W, the rest of column j (all GPs' first tiles, then their next)
        const int j = lo, at = (task - a.first[j] * a.batch) / a.batch, g = (task - a.first[j] * a.batch) % a.batch;
        const int diag = j >= a.i0 && j < T ? 1 : 0, wrow = j > a.i0 ? j - 1 : 0;
        double* Lg;
        double* Wg;
        double c[2][4][2] = {};
        if (at < diag || at >= diag + wrow) {
            const int i = at < diag ? j : max(j + 1, a.i0) + at - diag - wrow;
            int* lp = a.lprog + (size_t)g * T;
            Lg = a.L + (size_t)g * npad * npad;
            Wg = a.W + (size_t)g * npad * npad;
            gram_tile(a, g, i, j, smem, c);
            if (!accumulate<true>(a, g, i, j, 0, j, smem, sh, c)) return;
            __syncthreads();
            park(c, -1.0, tile0);
            __syncthreads();
            if (i == j) {
                factor_panel(tile0, 0, 2, tile1, sh.rinv, a, j * TB);
                __syncthreads();
                update_right(tile0, tile0, 32);
                __syncthreads();
                // one warp takes the second panel; the others hand the first one out meanwhile
                if (w == 0) {
                    factor_panel(tile0, 32, 1, tile1, sh.rinv, a, j * TB);
                } else {
                    store_half(Lg, npad, j, j, 0, tile0, t - 32, kThreads - 32, a.status);
                    asm volatile("bar.sync 2, 224;" ::: "memory");
                    if (t == 32 && announce) store_release_int(lp + j, 2 * j + 1);
                    for (int e = t - 32; e < 32 * 32; e += kThreads - 32) tile0[(e / 32) * kLd + 32 + e % 32] = 0.0;
                }
                __syncthreads();
                store_half(Lg, npad, j, j, 32, tile0, t, kThreads, a.status);
                publish(lp + j, 2 * j + 2, announce);
                for (int e = t; e < 32 * 32; e += kThreads) tile1[(e / 32) * kLd + 32 + e % 32] = 0.0;
                if (w < 2) invert_block(tile0, sh.rinv, 32 * w, tile1);
                __syncthreads();
                invert_corner(tile0, tile1, tile0);   // L11 is not needed any more
                store_tile(Wg, npad, j, j, tile1, a.status);
                publish(a.wprog + (size_t)g * T + j, 2 * j + 2);
            } else {
                // the left half against the first panel while the second is being made
                for (int h = 0; h < 64; h += 32) {
                    if (j >= a.i0 && !await(lp + j, 2 * j + 1 + h / 32)) return;
                    fetch_half(Lg, npad, j, h, tile1, a.status);
                    cp_async_wait<0>();
                    __syncthreads();
                    if (t < 32) sh.rinv[h + t] = 1.0 / tile1[(h + t) * kLd + h + t];
                    __syncthreads();
                    solve_panel(tile0, tile1, sh.rinv, h);
                    __syncthreads();
                    store_half(Lg, npad, i, j, h, tile0, t, kThreads, a.status);
                    publish(lp + i, 2 * j + 1 + h / 32, announce);
                    if (h == 0) update_right(tile0, tile1, 0);
                }
                zero_tile(Lg, npad, j, i, a.status);
                zero_tile(Wg, npad, j, i, a.status);
            }
        } else {
            const int i = j - 1, col = at - diag;
            Lg = a.L + (size_t)g * npad * npad;
            Wg = a.W + (size_t)g * npad * npad;
            int* wp = a.wprog + (size_t)g * T;
            if (!accumulate<false>(a, g, i, col, col, i, smem, sh, c)) return;
            if (!await(wp + i, 2 * i + 2)) return;
            fetch_tile(Wg, npad, i, i, tile0, a.status);
            park(c, -1.0, tile1);
            cp_async_wait<0>();
            __syncthreads();
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) c[p][q][0] = c[p][q][1] = 0.0;
#pragma unroll 1
            for (int k = 0; k < TB; k += 16)
                mma_step<false>(tile0 + (wm + l / 4) * kLd + k + l % 4, kLd, tile1 + (k + l % 4) * kLd + wn + l / 4, kLd, c);
            __syncthreads();
            park(c, 1.0, tile0);
            __syncthreads();
            store_tile(Wg, npad, i, col, tile0, a.status);
            publish(wp + col, 2 * i + 2);
        }
    }
}

// Clears the progress counters and looks the inputs over: non-finite values of X and y, min y and max |y| of every GP.
__global__ void __launch_bounds__(256) fit_begin_kernel(const float* __restrict__ X, size_t xcount, const float* __restrict__ y,
                                                        int n, float* __restrict__ best, float* __restrict__ yabs,
                                                        int* __restrict__ zero, int zeros, int* __restrict__ status)
{
    const int g = blockIdx.y;
    bool bad = false;
    const size_t step = (size_t)gridDim.x * gridDim.y * 256, at = ((size_t)g * gridDim.x + blockIdx.x) * 256 + threadIdx.x;
    for (size_t i = at; i < xcount; i += step) bad |= !isfinite(X[i]);
    for (size_t i = at; i < (size_t)zeros; i += step) zero[i] = 0;
    if (blockIdx.x == 0) {
        __shared__ float s[8], m[8];
        float v = INFINITY, u = 0.f;
        for (int i = threadIdx.x; i < n; i += 256) {
            const float yi = y[(size_t)g * n + i];
            bad |= !isfinite(yi);
            v = fminf(v, yi);
            u = fmaxf(u, fabsf(yi));
        }
        for (int o = 16; o > 0; o >>= 1) {
            v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
            u = fmaxf(u, __shfl_xor_sync(0xffffffffu, u, o));
        }
        if (threadIdx.x % 32 == 0) {
            s[threadIdx.x / 32] = v;
            m[threadIdx.x / 32] = u;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < 8; ++i) {
                v = fminf(v, s[i]);
                u = fmaxf(u, m[i]);
            }
            best[g] = v;
            yabs[g] = u;
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, DEV_NONFINITE);
}

}  // namespace

size_t factor_scratch_bytes(int batch, int npad)
{
    const size_t T = (npad + TB - 1) / TB;
    return sizeof(int) * (2 * (size_t)batch * T + 1);
}

r3_status_t factor_device(const FactorProblem& p, void* scratch, int extra_ints, int* status, int device, cudaStream_t stream)
{
    FactorArgs a;
    a.X = p.X; a.ell = p.ell; a.sf2 = p.sf2; a.sn2 = p.sn2;
    a.batch = p.batch; a.n = p.n; a.d = p.d; a.npad = p.npad;
    a.T = (p.npad + TB - 1) / TB;
    a.i0 = p.rows_done / TB;
    a.L = p.L; a.W = p.W;
    a.ticket = reinterpret_cast<unsigned*>(scratch);
    a.lprog = reinterpret_cast<int*>(scratch) + 1;
    a.wprog = a.lprog + (size_t)p.batch * a.T;
    a.status = status;
    a.wait = p.wait;
    a.first[0] = 0;
    for (int j = 0; j <= a.T; ++j)   // column j of L below the finished rows, row j - 1 of W
        a.first[j + 1] = a.first[j] + (j < a.T ? a.T - std::max(j, a.i0) : 0) + (j > a.i0 ? j - 1 : 0);
    const size_t xcount = (size_t)p.batch * p.n * p.d;
    const int zeros = (int)(factor_scratch_bytes(p.batch, p.npad) / sizeof(int)) + extra_ints;
    const unsigned gx = (unsigned)std::max<size_t>(1, std::min<size_t>(148, (xcount + 2047) / 2048) / p.batch);
    R3_LAUNCH(fit_begin_kernel, dim3(gx, p.batch), 256, 0, stream, p.X, xcount, p.y, p.n, p.best, p.yabs,
              reinterpret_cast<int*>(scratch), zeros, status);
    int sms = 148;
    R3_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    R3_CUDA_TRY(cudaFuncSetAttribute(factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFactorSmem));
    const long long tasks = (long long)a.first[a.T + 1] * a.batch;
    const unsigned grid = (unsigned)std::min<long long>(tasks, 2ll * sms);
    void* params[] = {&a};
    R3_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)factor_kernel, dim3(grid), dim3(kThreads), params, kFactorSmem, stream));
    ++g_launches;
    return R3_OK;
}

}  // namespace r3

extern "C" r3_status_t r3_test_rsqrt(const double* p, double* y, long long count, void* cuda_stream)
{
    using namespace r3;
    if (!p || !y || count < 1 || count >= (1ll << 31)) {
        set_error("r3_test_rsqrt: need two arrays and 1 <= count < 2^31");
        return R3_ERR_INVALID_ARG;
    }
    R3_LAUNCH(rsqrt_kernel, (unsigned)((count + 255) / 256), 256, 0, (cudaStream_t)cuda_stream, p, y, count);
    return R3_OK;
}
