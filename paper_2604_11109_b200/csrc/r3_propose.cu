// Greedy batch proposal by fantasies ("parallel" search of Section IV: several points of one search are
// replayed at once).  Definition: q times -- pick the not-yet-picked candidate of largest EI (incumbent
// fixed at the best observed value), then condition the GP on that point with a fantasised value (its
// posterior mean, "believer", or the incumbent, "liar").
//
// Refitting and rescoring the pool q times would cost q full scoring passes.  Conditioning on one point
// is a rank-one change of the posterior:
//     c(x) = cov(x, x_t),  s = var(x_t) + noise,
//     mu(x) += c(x) (value - mu(x_t)) / s,     var(x) -= c(x)^2 / s,
//     cov(x, x_t) = C0(x, x_t) - sum_{earlier picks u} c_u(x) c_u(x_t) / s_u,   C0(x, z) = k(x, z) - v(x).v(z),  v = W k*
// and with the believer's value the means never move while the variances only shrink, so EI (fixed
// incumbent) only drops: a candidate outside the R best of the first scoring can be picked only if some
// pick's EI falls below the (R+1)-th initial EI.  So: one full scoring with its top-(R+1), then the q picks on the
// shortlist alone, in FP64, in two kernels:
//   build_kernel  (cooperative) k* of the shortlist and k(z, z') of its pairs, which depend on nothing and are made together;
//                 then V = W k*; then C0 = k - V V^T; the products as tiles on the FP64 tensor path;
//   pick_kernel   (one cluster per GP) the q picks: a candidate per thread and part, the columns c_u in shared memory, one
//                 cluster barrier per pick.
// Bound: R n^2 / 2 + R^2 n / 2 FP64 multiply-adds, then the latency of a pick.  One GP of 4096 observations, 1023
// shortlisted, 128 picks: 6.1 ms as 259 launches (R n multiply-adds per pick), 1.8 ms now; 72 observations, 256
// shortlisted, 8 picks: 100 us in 19 launches and 46 us (62 us with k(z, z') made beside V V^T, after the second barrier).
#include <cooperative_groups.h>

#include <algorithm>

#include "r3_cross.cuh"
#include "r3_epilogue.cuh"
#include "r3_internal.cuh"

namespace r3 {

namespace {

namespace cg = cooperative_groups;

// All GPs of the handle are processed together; the shortlist state of GP g starts at g times the per-GP stride of each
// array.
struct ProposeArrays {
    const float* X;        // [B][n][d]
    const float* ell;      // [B][d]
    const float* sf2;      // [B]
    const float* sn2;      // [B]
    const float* best;     // [B]
    const double* alpha;   // [B][npad]
    const double* W;       // [B][npad][npad]
    const float* Xcand;    // [B][m][d]
    const int* sidx;       // [B][Rk] shortlist (pool indices), Rk >= R
    const float* sval;     // [B][Rk] their EI in the scoring of the pool
    long long m;
    int B, n, d, npad, R, Rk, q;
    double *Ks, *V;        // [B][R][npad]
    double *C0;            // [B][R][R] posterior covariances
    double *mupart;        // [B][R][ceil(npad / 64)]
    double *qpart;         // [B][R][ceil(npad / 64)]
    double *C;             // [B][q][R] columns of picks that do not fit shared memory
    int *cert;             // [B] the shortlist is certified to lose nothing
    unsigned* barrier;     // grid barrier, zero on entry
    int* status;
    WaitRule wait;
};

__device__ __forceinline__ const float* short_row(const ProposeArrays& a, int g, int r)
{
    return r < a.R ? a.Xcand + ((size_t)g * a.m + R3_IDX(a.sidx[(size_t)g * a.Rk + r], a.m, a.status)) * a.d : nullptr;
}

__global__ void __launch_bounds__(kCrossThreads, 2) build_kernel(const ProposeArrays a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int t = threadIdx.x, w = t / 32, l = t % 32, wm = (w % 4) * 16, wn = (w / 4) * 32;
    const int npad = a.npad, R = a.R, RT = (R + 63) / 64, NT = (npad + 63) / 64;
    unsigned target = 0;
    // ---- k* and the partial means; k(z, z') of the shortlist's own pairs, tiles (ta, tb) of the lower triangle
    const int pairs = RT * (RT + 1) / 2, kstar = a.B * RT * NT;
    auto pair_tile = [&](int p, int& ta, int& tb) {
        ta = 0;
        while ((ta + 1) * (ta + 2) / 2 <= p) ++ta;
        tb = p - ta * (ta + 1) / 2;
    };
    for (int item = blockIdx.x; item < kstar + (a.q > 1 ? a.B * pairs : 0); item += gridDim.x) {
        if (item < kstar) {
            const int g = item / (RT * NT), rt = item % (RT * NT) / NT, kb = item % NT;
            double* Ks = a.Ks + ((size_t)g * R + rt * 64) * npad;
            cross_tile<64>(
                a.n, a.d, npad, a.ell + (size_t)g * a.d, (double)a.sf2[g], a.alpha + (size_t)g * npad,
                [&](int r) { return short_row(a, g, rt * 64 + r); }, [&](int k) { return a.X + ((size_t)g * a.n + R3_IDX(k, a.n, a.status)) * a.d; }, kb,
                smem, [&](int c, int k, double v) { if (rt * 64 + c < R) Ks[(size_t)c * npad + R3_IDX(k, npad, a.status)] = v; },
                [&](int c, double s) { if (rt * 64 + c < R) a.mupart[((size_t)g * R + rt * 64 + c) * NT + kb] = s; });
        } else {
            const int g = (item - kstar) / pairs;
            int ta, tb;
            pair_tile((item - kstar) % pairs, ta, tb);
            double* C0 = a.C0 + (size_t)g * R * R;
            cross_tile<64>(
                R, a.d, R, a.ell + (size_t)g * a.d, (double)a.sf2[g], nullptr, [&](int r) { return short_row(a, g, ta * 64 + r); },
                [&](int k) { return short_row(a, g, k); }, tb, smem,
                [&](int r, int k, double v) { if (ta * 64 + r < R) C0[(size_t)(ta * 64 + r) * R + R3_IDX(k, R, a.status)] = v; }, [](int, double) {});
        }
    }
    if (!grid_barrier(a.barrier, target, a.status, a.wait)) return;
    // ---- V[r][i] = sum_k Ks[r][k] W[i][k], the longest rows of W first, and the partial sums of squares
    for (int item = blockIdx.x; item < a.B * RT * NT; item += gridDim.x) {
        const int it = NT - 1 - item / (a.B * RT), g = item % (a.B * RT) / RT, rt = item % RT;
        double c[2][4][2] = {};
        nt_tile(a.Ks + ((size_t)g * R + rt * 64) * npad, R - rt * 64, a.W + ((size_t)g * npad + it * 64) * npad, npad - it * 64,
                npad, min(npad, it * 64 + 64), smem, c, a.status);
        double* red = reinterpret_cast<double*>(smem);   // [2 column warps][64 rows]
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = rt * 64 + wm + 8 * i + l / 4;
            double s = 0.0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int col = it * 64 + wn + 8 * j + 2 * (l % 4);
                s = fma(c[i][j][0], c[i][j][0], fma(c[i][j][1], c[i][j][1], s));
                if (r < R && col < npad)
                    *reinterpret_cast<double2*>(a.V + ((size_t)g * R + r) * npad + col) = make_double2(c[i][j][0], c[i][j][1]);
            }
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (l % 4 == 0) red[(w / 4) * 64 + wm + 8 * i + l / 4] = s;
        }
        __syncthreads();
        if (t < 64 && rt * 64 + t < R) a.qpart[((size_t)g * R + rt * 64 + t) * NT + it] = red[t] + red[64 + t];
        __syncthreads();
    }
    if (a.q < 2) return;
    if (!grid_barrier(a.barrier, target, a.status, a.wait)) return;
    // ---- C0 = k(z, z') - V V^T, written on both sides
    for (int item = blockIdx.x; item < a.B * pairs; item += gridDim.x) {
        const int g = item / pairs;
        int ta, tb;
        pair_tile(item % pairs, ta, tb);
        const double* Vg = a.V + (size_t)g * R * npad;
        double* C0 = a.C0 + (size_t)g * R * R;
        double c[2][4][2] = {}, k0[2][4][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int row = ta * 64 + wm + 8 * i + l / 4, col = tb * 64 + wn + 8 * j + 2 * (l % 4) + h;
                    k0[i][j][h] = row < R && col < R ? __ldcg(C0 + (size_t)row * R + col) : 0.0;
                }
        nt_tile(Vg + (size_t)ta * 64 * npad, R - ta * 64, Vg + (size_t)tb * 64 * npad, R - tb * 64, npad, npad, smem, c, a.status);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int row = ta * 64 + wm + 8 * i + l / 4, col = tb * 64 + wn + 8 * j + 2 * (l % 4) + h;
                    if (row >= R || col >= R) continue;
                    const double v = k0[i][j][h] - c[i][j][h];
                    C0[(size_t)row * R + col] = v;
                    if (ta != tb) C0[(size_t)col * R + row] = v;
                }
    }
}

constexpr int kPickThreads = 1024;
constexpr int kMaxCluster = 8;
constexpr int kMaxPicks = 256;
struct Best {
    unsigned long long key;   // bits of the EI plus one, 0: no candidate
    int idx, r;               // pool index, place in the shortlist
    double mu, var;
};
struct PickShared {
    Best slot[2][kMaxCluster];
    Best warp_best[kPickThreads / 32];
    double w[kMaxPicks], inv_s[kMaxPicks], part[kPickThreads];
};
constexpr size_t kPickSmem = 224 * 1024;

__device__ __forceinline__ bool better(unsigned long long ka, int ia, unsigned long long kb, int ib)
{
    return ka > kb || (ka == kb && ia < ib);   // equal EI: the lower pool index
}

// One cluster per GP, the shortlist cut into one piece of Rl candidates per block; `held` columns c_u in shared memory.
__global__ void __launch_bounds__(kPickThreads, 1) pick_kernel(const ProposeArrays a, int liar, int Rl, int held,
                                                               int* __restrict__ idx_all, float* __restrict__ ei_all)
{
    extern __shared__ __align__(16) unsigned char smem[];
    PickShared& sh = *reinterpret_cast<PickShared*>(smem);
    double* cols = reinterpret_cast<double*>(smem + sizeof(PickShared));   // [held][Rl]
    cg::cluster_group cluster = cg::this_cluster();
    const int CS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int g = blockIdx.x / CS, t = threadIdx.x, lane = t % 32, warp = t / 32;
    const int R = a.R, NT = (a.npad + 63) / 64;
    const int parts = kPickThreads / Rl, part = t / Rl, mine = t % Rl;   // Rl is a multiple of 32
    const int r = rank * Rl + mine;
    const bool active = part < parts && r < R, owner = active && part == 0;
    const double best = (double)a.best[g], sn2 = (double)a.sn2[g];
    const double* C0 = a.C0 + (size_t)g * R * R;
    double* Cg = a.C + (size_t)g * a.q * R;
    double mu = 0.0, var = 0.0;
    int idx = 0;
    bool picked = true;
    if (owner) {
        double s = 0.0;
        for (int b = 0; b < NT; ++b) {
            mu += a.mupart[((size_t)g * R + r) * NT + b];
            s += a.qpart[((size_t)g * R + r) * NT + b];
        }
        var = (double)a.sf2[g] - s;
        idx = a.sidx[(size_t)g * a.Rk + r];
        picked = false;
    }
    double lowest = INFINITY;
    for (int step = 0; step < a.q; ++step) {
        // ---- the largest EI of the block, then of the cluster
        Best m = {0ull, 0x7fffffff, 0, 0.0, 0.0};
        if (owner && !picked) {
            const double ei = ei_closed_form(mu, sqrt(fmax(var, 0.0)), best), e = ei >= 0.0 ? ei : 0.0;   // NaN counts as 0
            m = {(unsigned long long)__double_as_longlong(e) + 1ull, idx, r, mu, var};   // e >= 0
        }
        unsigned long long key = m.key;
        int who = m.idx, from = lane;
        if (warp * 32 < Rl) {
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
                const int i2 = __shfl_xor_sync(0xffffffffu, who, o), f2 = __shfl_xor_sync(0xffffffffu, from, o);
                if (better(k2, i2, key, who)) {
                    key = k2;
                    who = i2;
                    from = f2;
                }
            }
            if (lane == from) sh.warp_best[warp] = m;
        }
        __syncthreads();
        if (warp == 0) {
            m = lane < Rl / 32 ? sh.warp_best[lane] : Best{0ull, 0x7fffffff, 0, 0.0, 0.0};
            key = m.key;
            who = m.idx;
            from = lane;
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
                const int i2 = __shfl_xor_sync(0xffffffffu, who, o), f2 = __shfl_xor_sync(0xffffffffu, from, o);
                if (better(k2, i2, key, who)) {
                    key = k2;
                    who = i2;
                    from = f2;
                }
            }
            if (lane == from)
                for (int b = 0; b < CS; ++b) *cluster.map_shared_rank(&sh.slot[step & 1][rank], b) = m;
        }
        cluster.sync();
        Best win = sh.slot[step & 1][0];
        for (int b = 1; b < CS; ++b)
            if (better(sh.slot[step & 1][b].key, sh.slot[step & 1][b].idx, win.key, win.idx)) win = sh.slot[step & 1][b];
        const int j = win.r;
        const double e = __longlong_as_double((long long)(win.key - 1ull));
        double s = fmax(win.var, 0.0) + sn2, delta = 0.0;
        if (!(s > 0.0)) {   // a candidate on top of an observation with zero noise: nothing to condition on
            if (rank == 0 && t == 0) atomicOr(a.status, DEV_NOT_PD);
            s = INFINITY;
        } else {
            // the fantasised value enters the history as an observation, i.e. rounded to FP32
            const double value = liar ? best : (double)(float)win.mu;
            delta = (value - win.mu) / s;
        }
        lowest = fmin(lowest, (double)(float)e);
        if (rank == 0 && t == 0) {
            idx_all[(size_t)g * a.q + step] = win.idx;
            if (ei_all) ei_all[(size_t)g * a.q + step] = (float)e;
        }
        if (owner && r == j) picked = true;
        if (step + 1 == a.q) break;
        // ---- c(x) = C0(x, x_j) - sum_u c_u(x) c_u(x_j) / s_u
        double c = owner ? C0[(size_t)R3_IDX(j, R, a.status) * R + r] : 0.0;
        const int jr = j / Rl, jl = j % Rl;
        const double* theirs = cluster.map_shared_rank(cols, jr);
        for (int u = t; u < step; u += kPickThreads)
            sh.w[u] = (u < held ? theirs[R3_IDX((size_t)u * Rl + jl, (size_t)held * Rl, a.status)] : __ldcg(Cg + (size_t)u * R + j)) * sh.inv_s[u];
        if (t == 0) sh.inv_s[step] = 1.0 / s;
        __syncthreads();
        double s0 = 0.0, s1 = 0.0;
        if (active) {
            int u = part;
            for (; u + parts < step; u += 2 * parts) {
                const double x = u < held ? cols[(size_t)u * Rl + mine] : Cg[(size_t)u * R + r];
                const double y = u + parts < held ? cols[(size_t)(u + parts) * Rl + mine] : Cg[(size_t)(u + parts) * R + r];
                s0 = fma(x, sh.w[u], s0);
                s1 = fma(y, sh.w[u + parts], s1);
            }
            if (u < step) s0 = fma(u < held ? cols[(size_t)u * Rl + mine] : Cg[(size_t)u * R + r], sh.w[u], s0);
        }
        sh.part[t] = s0 + s1;
        __syncthreads();
        if (owner) {
            for (int p = 0; p < parts; ++p) c -= sh.part[p * Rl + mine];
            if (step < held) cols[R3_IDX((size_t)step * Rl + mine, (size_t)held * Rl, a.status)] = c;
            else Cg[(size_t)step * R + r] = c;
            mu = fma(c, delta, mu);
            var -= c * c / s;
        }
    }
    if (rank == 0 && t == 0) {
        // The believer's EI only drops: nothing outside the shortlist could have been picked while the picks stayed above
        // the best EI left out (FP32, within the scoring tolerance of 1e-5 max EI).
        int cert = 1;
        if (a.Rk > R) {
            const double bound = a.sval[(size_t)g * a.Rk + R], top = a.sval[(size_t)g * a.Rk];
            cert = !liar && lowest >= bound + 4e-5 * top ? 1 : 0;
        }
        a.cert[g] = cert;
    }
    cluster.sync();   // no block leaves while another may read its shared memory
}

size_t up16(size_t b) { return (b + 15) & ~(size_t)15; }

}  // namespace

size_t propose_workspace_bytes(int batch, int npad, int R, int q)
{
    const size_t B = batch, NT = (npad + 63) / 64;
    return up16(sizeof(double) * B * R * (2 * (size_t)npad + R + 2 * NT)) + up16(sizeof(double) * B * q * R) +
           up16(sizeof(int) * B) + 256;
}

// The q picks of every GP of the handle.  sidx, sval: device [batch][Rk] pool indices and EI of the shortlists (by initial
// EI, descending; the first R of each row are used); idx_out / ei_out: device [batch][q]; *cert: device [batch].
// ws: propose_workspace_bytes(batch, npad, R, q) bytes.
r3_status_t propose_shortlist(r3_gp* gp, const float* Xcand, long long m, const int* sidx, const float* sval, int Rk, int R,
                              int q, int liar, int* idx_out, float* ei_out, int** cert, void* ws, cudaStream_t stream)
{
    ProposeArrays a;
    a.X = gp->X; a.ell = gp->ell_d; a.sf2 = gp->sf2_d; a.sn2 = gp->sn2_d; a.best = gp->best_d; a.alpha = gp->alpha64;
    a.W = gp->W64; a.Xcand = Xcand; a.sidx = sidx; a.sval = sval;
    a.m = m;
    a.B = gp->batch; a.n = gp->n; a.d = gp->d; a.npad = gp->npad; a.R = R; a.Rk = Rk; a.q = q;
    const size_t B = a.B, npad = a.npad, NT = (npad + 63) / 64;
    a.Ks = (double*)ws;
    a.V = a.Ks + B * R * npad;
    a.C0 = a.V + B * R * npad;
    a.mupart = a.C0 + B * R * R;
    a.qpart = a.mupart + B * R * NT;
    char* p = (char*)ws + up16(sizeof(double) * B * R * (2 * npad + R + 2 * NT));
    a.C = (double*)p;
    p += up16(sizeof(double) * B * q * R);
    a.cert = (int*)p;
    p += up16(sizeof(int) * B);
    a.barrier = (unsigned*)p;
    a.status = gp->status_d;
    a.wait = wait_rule(gp, STALL_PROPOSE);
    *cert = a.cert;
    R3_CUDA_TRY(cudaMemsetAsync(a.barrier, 0, sizeof(unsigned), stream));

    int sms = 148;
    R3_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, gp->device));
    R3_CUDA_TRY(cudaFuncSetAttribute(build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCrossStageBytes));
    const long long RT = (R + 63) / 64, items = B * (RT * NT + RT * (RT + 1) / 2);   // of the first phase, the widest
    const unsigned grid = (unsigned)std::min<long long>(2ll * sms, items);
    void* params[] = {&a};
    R3_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)build_kernel, dim3(grid), dim3(kCrossThreads), params, kCrossStageBytes,
                                            stream));
    ++g_launches;

    // One block as long as its shared memory holds the columns of all picks, else a cluster of eight.  Whole proposals from
    // 4096 candidates (300 observations, 16 features), one block | eight: 16 picks from 256 259 | 271 us, 32 from 256 313 | 331,
    // 48 from 384 395 | 393, 56 from 448 455 | 428 (the last sizes that one block holds), 64 from 512 516 | 465, 128 from 1023
    // 1751 | 827.  With eight GPs side by side the differences are the same.
    const size_t room = (kPickSmem - sizeof(PickShared)) / sizeof(double);
    int CS = 1, Rl = round_up(R, 32);
    if ((size_t)Rl * (q - 1) > room) {
        CS = kMaxCluster;
        Rl = round_up((R + CS - 1) / CS, 32);
    }
    const int held = (int)std::min<size_t>(q, room / Rl);
    R3_CUDA_TRY(cudaFuncSetAttribute(pick_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPickSmem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(B * CS));
    cfg.blockDim = dim3(kPickThreads);
    cfg.dynamicSmemBytes = sizeof(PickShared) + sizeof(double) * (size_t)held * Rl;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    R3_CUDA_TRY(cudaLaunchKernelEx(&cfg, pick_kernel, a, liar, Rl, held, idx_out, ei_out));
    ++g_launches;
    return R3_OK;
}

}  // namespace r3
