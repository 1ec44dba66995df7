// Tensor-core scoring engine for sm_100a: tcgen05 MMAs (kind::f16 on two-term FP16 splits, FP32
// accumulation in TMEM), operands staged by bulk asynchronous copies, everything fused in one kernel
// so that the cross-covariance k* never leaves the SM.
//
// One CTA owns a tile of 128 candidates; a TMEM lane IS a candidate.  For that tile it walks the rows of W = L^-1 in strips
// of 128 (a V accumulator: 128 lanes x 128 TMEM columns) and, for a strip, the observations in chunks of KC = 32:
//
//   distance MMA   D[cand][k] = z~ . x~_k   (A = scaled candidates, B = scaled observations, both in shared memory, depth d),
//                  for 64 observations at a time
//   Matern warps   r^2 = |z~|^2 + |x~_k|^2 - 2 D, k* = sf2 M52(r): read D from TMEM and write k* (scaled, FP16 hi/lo planes)
//                  over it, where it is the next A operand; mu += k* alpha on the way
//   variance MMA   V[cand][i] += k*[cand][k] W[i][k]   (B = pre-tiled chunk of W, scaled FP16 hi/lo planes)
//   end of strip   q += sum_i V[cand][i]^2 read back from TMEM; after the last strip sigma, EI, outputs
//
// Precision.  Every product is three MMAs (hi*hi + hi*lo + lo*hi): x = hi + lo with hi = fp16(x) and
// lo = fp16(x - hi) carries 22 significant bits, and the tensor core accumulates in FP32, so the
// result is FP32-grade at twice the TF32 rate and half the operand bytes.  k* and W are multiplied by
// powers of two before the split (so that the low parts stay normal numbers) and the accumulator is
// scaled back exactly.  The scaled coordinates of the distance product must fit FP16's range; a
// history that does not is left to the SIMT engine and a candidate that does not is recomputed in FP64.
//
// W is lower-triangular, so strip s only needs k < 128 (s + 1).  Strips come in pairs that share the k* chunks; from pair to
// pair the chunks are generated again instead of being stored.
//
// What the layout is for: nothing waits for a whole pass or a whole tile.  The two accumulators are filled by issuers of their
// own, so that one is read back while the other's products run; the ring of eight k* slots and the second buffer of scaled
// candidates let the next pair's and the next tile's chunks be made meanwhile; candidates come in and results go out through
// warps of their own, not through the Matern warps.  TMEM: two accumulators (256 columns) and the ring (8 x 32), all 512.
// A tile of 512 observations and 32 features takes 33,000 cycles (48,700 as passes of 256 rows with one accumulator, whose
// Matern warps also brought the candidates in and read the accumulator back); its MMAs alone take 16,400.
//
// Warp roles: warp 0 streams the operands (three lanes: scaled observations, chunks of W for either accumulator), warp 1
// issues the distance MMAs, warps 2 and 3 the variance MMAs of one accumulator each (the issuing roles are whole warps, see
// mbar_wait_warp); two groups of four warps bring candidates in and results out; three groups of four Matern warps (one warp
// per TMEM lane quarter) take every third chunk each.  Stages are handed over through mbarriers; every wait is bounded: when
// a limit is hit the CTA raises a status bit, all roles leave their loops, in-flight copies and MMAs are drained (bounded
// again), TMEM is freed and the kernel returns.  Between set-up and teardown no warp waits for another in any other way: whether
// a wait ran out is decided by each warp for itself, so a barrier without a limit (bar.sync) could be entered by one warp of a
// group after another has left.  Warps of a group therefore share nothing but mbarriers: a warp finishes its own 32 rows,
// counts the parts of its own rows of a shared tile, and leaves its own largest EI.
//
// The roles' code has to stay small: together it is about what the SM's instruction cache holds, and what does not fit costs
// the Matern warps first.  Both halves of a chunk unrolled, norms and weights through shared memory (one more wait in the
// loop), waits with a long form of their time-out: each of them raised the cache's misses from 0.5 M to 1.4-1.7 M per million
// candidates' worth of tiles and the kernel's time by 19-27 % (64 pools of 65,536 candidates, 512 observations).
//
// Operand layouts are the no-swizzle K-major "core matrix" form: 8 rows x 16 bytes contiguous, 8-row
// groups 128 bytes apart, 16-byte k-slices one full panel apart.  W and the observations are stored
// in global memory already tiled that way by the fit, so a stage is one contiguous bulk copy.
#include <algorithm>
#include <cuda_fp16.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "r3_epilogue.cuh"
#include "r3_f32x2.cuh"
#include "r3_internal.cuh"
#include "r3_tc_common.cuh"

namespace r3 {

namespace {

constexpr int kStrip = 128;              // rows of W per accumulator
constexpr int kSlots = 8;                // ring of k* slots of KC tensor-memory columns
constexpr uint32_t kRingCol = 2 * kStrip;
constexpr int kMaxWS = 8, kMaxXS = 3;    // stages of W (half for each accumulator) and of scaled observations
constexpr int KDC = 2, KD = KDC * KC;    // chunks and observations per distance product, which fills a bank of slots
constexpr int BANKS = kSlots / KDC;
constexpr int IO = 2, G = 3;             // groups of four warps: candidates in and results out (one per buffer), Matern
constexpr int kFirstIo = 4, kFirstMatern = kFirstIo + 4 * IO, kThreads = kFirstMatern * 32 + 128 * G;
constexpr int kZ32MaxDP = 32;            // features up to which the scaled tile is kept in FP32 too
constexpr int kPartDP = 64;              // features per stage of scaled observations at most

// barrier slots (8 bytes each)
enum : uint32_t {
    BAR_X_FULL = 0, BAR_X_EMPTY = BAR_X_FULL + kMaxXS, BAR_W_FULL = BAR_X_EMPTY + kMaxXS, BAR_W_EMPTY = BAR_W_FULL + kMaxWS,
    BAR_D_FULL = BAR_W_EMPTY + kMaxWS, BAR_K_EMPTY = BAR_D_FULL + 4, BAR_K_FULL = BAR_K_EMPTY + 4,
    BAR_V_FULL = BAR_K_FULL + kSlots,   // [accumulator][group that reads it back]
    BAR_V_EMPTY = BAR_V_FULL + 4, BAR_Z_FULL = BAR_V_EMPTY + 2, BAR_Z_EMPTY = BAR_Z_FULL + 2,
    BAR_RED_FULL = BAR_Z_EMPTY + 2, BAR_RED_EMPTY = BAR_RED_FULL + 2, BAR_MMA_DONE = BAR_RED_EMPTY + 2,   // MMA_DONE: three, distance and variance issuers
    BAR_COUNT = BAR_MMA_DONE + 3
};
constexpr uint32_t kFlagOffset = 512;    // behind the barriers: int abort, int drain-abort, uint32 tmem base
static_assert(BAR_COUNT * 8 <= kFlagOffset, "barriers overlap the flags");
constexpr uint32_t kBarBytes = 1024;
// Registers per thread once the roles have parted; the block starts with the file split evenly (80 for 768 threads).
// The forms without FP8 cross terms spill nothing with this split (88 for the Matern warps and 80 for results: 20 bytes); those
// with them spill five to eight registers, no fewer with any other split (64/72/88: ten and four) nor with the two halves of a
// chunk's dot products read one after the other.
constexpr int kRegsControl = 48, kRegsIo = 72, kRegsMatern = 96;
static_assert(kRegsControl + IO * kRegsIo + G * kRegsMatern <= 80 * (kThreads / 128), "more registers than the block starts with");

// per buffer of scaled candidates: float[128] squared norms, float[128] thresholds of close pairs, then the tile's scale of
// k*, 1 / (the power of two in it) and GP
constexpr uint32_t kZnBuf = TILE_M * 8u + 16u;

// shared-memory map (byte offsets from a 1024-aligned base)
struct SmemMap {
    uint32_t z, z32, x, w, red, zn, cache, bar, end;
    uint32_t z_buf, z32_buf, red_buf, x_stage;
};
__host__ __device__ inline SmemMap smem_map(int DP, int parts, int zb, int xs, int ws)
{
    SmemMap s;
    s.z_buf = 512u * DP;                                  // scaled candidates: FP16 hi plane, lo plane, [DP/8][128][8] each
    s.z32_buf = DP <= kZ32MaxDP ? 512u * DP : 0u;         // the same in FP32, [DP/4][128][4]
    s.x_stage = 4u * (DP / parts) * KD;                   // scaled observations: two planes [DP/parts/8][KD][8]
    s.z = 0;
    s.z32 = s.z + zb * s.z_buf;
    s.x = s.z32 + zb * s.z32_buf;
    s.w = s.x + xs * s.x_stage;                           // chunks of W: two planes [KC/8][rows][8]
    s.red = s.w + ws * (4u * KC * kStrip);                // mu and two error scales of each group and row, doubles
    s.red_buf = 3u * G * TILE_M * 8u;
    s.zn = s.red + zb * s.red_buf;            // see kZnBuf
    s.cache = s.zn + 2u * kZnBuf;                    // refined close pairs of the tile (see refine_close_pairs)
    s.bar = s.cache + (DP <= kZ32MaxDP ? 0u : TILE_M * kCacheSlots * 8u);
    s.end = s.bar + kBarBytes;
    return s;
}

// a - h exactly, in one mixed-precision instruction
__device__ __forceinline__ float minus_half(float a, __half h)
{
    float r;
    asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(r) : "h"(__half_as_ushort(h)), "h"((unsigned short)0xbc00), "f"(a));
    return r;
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t* r)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
                 "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                 "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
                 : "memory");
}

// The strips (128 rows of W) of a tile come in pairs that share the k* chunks.  Strip a = 2 p needs the first `na` chunks of
// the history, strip a + 1, where there is one, the first `nb`.
struct Pair {
    int a, na, nb;   // nb = 0: a single strip
    __device__ __forceinline__ Pair(int p, int S, int nc) : a(2 * p), na(min(4 * (a + 1), nc)), nb(a + 1 < S ? min(4 * (a + 2), nc) : 0) {}
    __device__ __forceinline__ int chunks() const { return nb ? nb : na; }
};

// Waits and issue for a role that is a whole warp: every lane takes the same path, so that operand addresses and descriptors
// are computed on the uniform datapath (a role of one lane spent 450 cycles per chunk moving them there, as long as the
// products took); the instructions that one thread has to issue are predicated on the elected lane.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, long long limit)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    do {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    } while (!__any_sync(0xffffffffu, (*abort_flag != 0) | (clock64() - t0 > limit)));
    *abort_flag = 1;
    return false;
}
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r;
}
__device__ __forceinline__ void tc_commit_if(uint32_t leader, uint32_t bar)
{
    asm volatile(
        "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %1, 0;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(leader)
        : "memory");
}
__device__ __forceinline__ void tc_mma_f16_if(uint32_t leader, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc),
        "r"(accumulate), "r"(leader)
        : "memory");
}
__device__ __forceinline__ void tc_mma_f16_ts_if(uint32_t leader, uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc),
        "r"(accumulate), "r"(leader)
        : "memory");
}
__device__ __forceinline__ void tc_mma_f8_ts_if(uint32_t leader, uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc),
        "r"(accumulate), "r"(leader)
        : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Close pairs of a candidate row with the scaled tile in shared memory as FP16 planes: k* recomputed from direct differences.
// Out of line; per lane, one pair at a time.  z: this row's 16 bytes of the first slice of the hi plane.
__device__ __noinline__ void refine_close_pairs_smem(float* kv, float v_thresh, float kvscale, const uint8_t* z, int DP,
                                                     const float* __restrict__ xrow0, unsigned long long* slots, uint32_t key0,
                                                     bool lookup)
{
    uint32_t close = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) close |= (kv[i] > v_thresh) ? (1u << i) : 0u;
    const uint32_t lo_plane = 256u * DP;
    for (uint32_t rest = close; rest; rest &= rest - 1) {
        const int i = __ffs(rest) - 1;
        if (slots && lookup) {
            const unsigned long long e = slots[cache_slot(key0 + i)];
            if ((uint32_t)(e >> 32) == key0 + i) {
                kv[i] = __uint_as_float((uint32_t)e);
                continue;
            }
        }
        const float4* xp = reinterpret_cast<const float4*>(xrow0 + (size_t)i * DP);
        float acc0 = 0.f, acc1 = 0.f;
#pragma unroll 2
        for (int j8 = 0; j8 < DP / 8; ++j8) {
            const uint4 zh = *reinterpret_cast<const uint4*>(z + j8 * 2048u);
            const uint4 zl = *reinterpret_cast<const uint4*>(z + lo_plane + j8 * 2048u);
            const float4 xa = __ldg(xp + 2 * j8), xb = __ldg(xp + 2 * j8 + 1);
            const float x[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
            const uint32_t h[4] = {zh.x, zh.y, zh.z, zh.w}, l[4] = {zl.x, zl.y, zl.z, zl.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&h[e]));
                const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&l[e]));
                float df = (a.x + b.x) - x[2 * e];
                acc0 = fmaf(df, df, acc0);
                df = (a.y + b.y) - x[2 * e + 1];
                acc1 = fmaf(df, df, acc1);
            }
        }
        const float u = sqrtf(acc0 + acc1);
        kv[i] = kvscale * fmaf(u, fmaf(u, kPolyC2, kPolyC1), 1.f) * exp2f(-u);
        if (slots) slots[cache_slot(key0 + i)] = ((unsigned long long)(key0 + i) << 32) | __float_as_uint(kv[i]);
    }
}

// F8: the two cross terms of the variance product (W_hi k_lo, W_lo k_hi) are single FP8 MMAs of depth 32 instead of two FP16
// MMAs of depth 16 each: four MMAs per chunk and strip instead of six.
// Z32: at most 32 features: the scaled candidates are also kept in FP32 and close pairs are refined inline from them (pools of
// few features are full of close pairs: on 16 features 98 % of a warp's 16-entry blocks hold one).
// FEW: at most 16 features (with Z32): many entries of a block are close at once and a row of observations is short.  Refined values
// go through a local array instead of a selection among sixteen each, and up to 8 features the padding is passed over.  58,087
// candidates, 1779 observations, 3 features, all of which FP64 recomputes afterwards: whole call 11.66 -> 10.91 ms; 100,000, 400, 9:
// 0.438 -> 0.406 ms; 262,144, 256, 16: 0.214 -> 0.210 ms.  With 17 to 32 features few entries are close at once and the local array
// costs more than the selections (199,999, 701, 23: 0.682 -> 0.765 ms).
template <bool F8, bool Z32, bool FEW>
__global__ void __launch_bounds__(kThreads, 1) score_tc_kernel(const __grid_constant__ TcParams prm)
{
    if (prm.mode && *prm.mode != prm.want_mode) return;   // the other form of the kernel serves this pool
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - raw);
    const int DP = prm.DP, parts = prm.parts, DPp = DP / parts, nc = prm.nc, S = prm.S;
    const int zb = prm.zb, xs = prm.xs, ws = prm.ws;
    const SmemMap map = smem_map(DP, parts, zb, xs, ws);
    const uint32_t bars = base + map.bar;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + map.bar + kFlagOffset);
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + map.bar + kFlagOffset + 8);
    auto zn_buf = [&](int b) { return reinterpret_cast<float*>(sm + map.zn + b * kZnBuf); };
    auto bar = [&](uint32_t slot) { return bars + slot * 8u; };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t TMEM_COLS = 512u;
    const long long wl = prm.wait_limit;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kMaxXS; ++i) {
            mbar_init(bar(BAR_X_FULL + i), 1);
            mbar_init(bar(BAR_X_EMPTY + i), 1);
        }
        for (int i = 0; i < kMaxWS; ++i) {
            mbar_init(bar(BAR_W_FULL + i), 1);
            mbar_init(bar(BAR_W_EMPTY + i), 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(bar(BAR_D_FULL + i), 1);
            mbar_init(bar(BAR_K_EMPTY + i), 2);
        }
        for (int i = 0; i < kSlots; ++i) mbar_init(bar(BAR_K_FULL + i), 4);
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(BAR_V_FULL + i), 1);
            mbar_init(bar(BAR_V_FULL + 2 + i), 1);
            mbar_init(bar(BAR_V_EMPTY + i), 4);
            mbar_init(bar(BAR_RED_FULL + i), 4 * G);
            mbar_init(bar(BAR_RED_EMPTY + i), 4);
            mbar_init(bar(BAR_Z_FULL + i), 4);
            mbar_init(bar(BAR_Z_EMPTY + i), 1 + 4 * G);
        }
        for (int i = 0; i < 3; ++i) mbar_init(bar(BAR_MMA_DONE + i), 1);
        abort_flag[0] = 0;
        abort_flag[1] = 0;   // private flag of the bounded drain waits
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (!Z32) {
        unsigned long long* pair_cache = reinterpret_cast<unsigned long long*>(sm + map.cache);
        for (int i = threadIdx.x; i < TILE_M * (int)kCacheSlots; i += blockDim.x) pair_cache[i] = ~0ull;   // a key that no (tile, observation) forms
    }
    // the guard's counters (with FP8 cross terms the pilot clears them)
    if constexpr (!F8)
        if (blockIdx.x == 0)
            for (int i = threadIdx.x; i < prm.zero_ints; i += blockDim.x) prm.zero[i] = 0;
    if (warp == 2) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32((const void*)tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // units of this CTA: blockIdx.x, blockIdx.x + gridDim.x, ...; a unit is the pairs [cut[part], cut[part + 1]) of a tile
    const int tiles = (int)(prm.total_tiles - prm.tile_begin), units = tiles * prm.splits, unit_step = (int)gridDim.x;
    const uint32_t tiles_per_gp = (uint32_t)prm.tiles_per_gp;
    auto part_of = [&](int unit) { return prm.splits == 1 ? 0 : prm.splits - 1 - (int)((uint32_t)unit / (uint32_t)tiles); };   // the longest parts first
    auto tile_of = [&](int unit) { return (uint32_t)prm.tile_begin + (prm.splits == 1 ? (uint32_t)unit : (uint32_t)unit % (uint32_t)tiles); };

    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsControl));
    const uint32_t leader = elect_one();
    if (warp == 0) {
        // ------------------------------------------------------------ producer: three lanes, a stream each
        // lane 0: scaled observations; lanes 1 and 2: the chunks of W of the strips that go to accumulator 0 and 1.  The lanes
        // poll together, so that no stream waits for another.
        const int me = lane - 1, ring = lane == 0 ? xs : ws / 2;
        const uint32_t full0 = lane == 0 ? BAR_X_FULL : BAR_W_FULL + me * (kMaxWS / 2), empty0 = lane == 0 ? BAR_X_EMPTY : BAR_W_EMPTY + me * (kMaxWS / 2);
        const uint32_t dst0 = base + (lane == 0 ? map.x : map.w + me * ring * (4u * KC * kStrip)), stride = lane == 0 ? map.x_stage : 4u * KC * kStrip;
        long long issued = 0;
        int st = 0, unit = blockIdx.x, p = 0, strip = 0, strips = 0, c = 0, count = 0;
        uint32_t ph = 0, bytes = 0, sigma = 0;
        const __half* src = nullptr;
        bool have = lane < 3 && unit < units;
        int p_end = 0, g = 0;
        auto open_unit = [&] {
            const int part = part_of(unit);
            p = prm.cut[part];
            p_end = prm.cut[part + 1];
            g = (int)(tile_of(unit) / tiles_per_gp);
        };
        if (have) open_unit();
        auto next_segment = [&] {   // the next run of equal blobs: a pair's observations, or the chunks of one of its strips
            c = 0;
            while (have) {
                if (strip == strips) {   // next pair
                    if (strips && ++p == p_end) {
                        if ((unit += unit_step) >= units) { have = false; break; }
                        open_unit();
                    }
                    strip = 0;
                    strips = lane == 0 || !Pair(p, S, nc).nb ? 1 : 2;
                }
                const Pair pr(p, S, nc);
                const int s = pr.a + strip++;
                if (lane == 0) {
                    src = prm.xt + (size_t)g * prm.NP * 2 * DP;
                    count = pr.chunks() / KDC * parts;
                    bytes = map.x_stage;
                    break;
                }
                if ((int)(sigma++ & 1u) == me) {
                    const int rows = min(kStrip, nc * KC - s * kStrip);
                    src = prm.wt + (size_t)g * prm.wt_gp_stride +
                          R3_IDX((size_t)2 * s * (s + 1) * (2 * KC * kStrip), prm.wt_gp_stride, prm.status);
                    count = min(4 * (s + 1), nc);
                    bytes = 4u * KC * rows;
                    break;
                }
            }
        };
        next_segment();
        bool ok = true;
        long long t0 = clock64();
        while (__any_sync(0xffffffffu, have)) {
            const bool held = lane == 1 && issued == prm.withhold_w;   // test aid: this stream of W stops here
            bool moved = false;
            if (have && !held && mbar_test(bar(empty0 + st), ph ^ 1u)) {
                mbar_arrive_expect_tx(bar(full0 + st), bytes);
                bulk_g2s(dst0 + (uint32_t)R3_IDX(st, ring, prm.status) * stride, src + (size_t)c * (bytes / 2), bytes, bar(full0 + st));
                ++issued;
                if (++st == ring) { st = 0; ph ^= 1u; }
                if (++c == count) next_segment();
                moved = true;
            }
            if (__any_sync(0xffffffffu, moved)) {
                t0 = clock64();
                continue;
            }
            if (__any_sync(0xffffffffu, *abort_flag)) { ok = false; break; }
            if (__any_sync(0xffffffffu, clock64() - t0 > wl)) {
                *abort_flag = 1;
                ok = false;
                break;
            }
            __nanosleep(100);
        }
        if (!ok && lane < 3) {  // aborting: let the copies still in flight land before the CTA goes away
            const int pending = (int)(issued < ring ? issued : ring);
            for (int u = 0; u < pending; ++u) {
                if (--st < 0) { st = ring - 1; ph ^= 1u; }
                mbar_wait(bar(full0 + st), ph, abort_flag + 1, wl);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: distance products
        constexpr uint32_t IDESC_D = instr_desc_f16(KD);
        // descriptor low word = start >> 4 | (k-slice distance >> 4) << 16
        const uint32_t z_lo0 = desc_addr(base + map.z) | ((2048u >> 4) << 16);
        const uint32_t x_lo0 = desc_addr(base + map.x) | (((KD * 16u) >> 4) << 16);
        const int ksteps = DPp / 16;
        const uint32_t x_plane = ((uint32_t)DPp * KD * 2u) >> 4, z_plane = (256u * DP) >> 4;
        int st = 0, bank = 0, zi = 0;
        uint32_t ph = 0, bank_ph = 0, z_ph = 0;
        bool ok = true;
        for (int unit = blockIdx.x; ok && unit < units; unit += unit_step) {
            const int part = part_of(unit);
            if (!(ok = mbar_wait_warp(bar(BAR_Z_FULL + zi), z_ph, abort_flag, wl))) break;
            tc_fence_after();
            for (int p = prm.cut[part]; ok && p < prm.cut[part + 1]; ++p) {
                const int products = Pair(p, S, nc).chunks() / KDC;
                for (int u = 0; ok && u < products; ++u) {
                    if (!(ok = mbar_wait_warp(bar(BAR_K_EMPTY + bank), bank_ph ^ 1u, abort_flag, wl))) break;
                    const uint32_t dcol = tmem + kRingCol + (uint32_t)R3_IDX(bank, BANKS, prm.status) * KD;
                    uint32_t acc = 0;
                    for (int q = 0; q < parts; ++q) {
                        if (!(ok = mbar_wait_warp(bar(BAR_X_FULL + st), ph, abort_flag, wl))) break;
                        tc_fence_after();
                        const uint32_t xH = x_lo0 + ((st * map.x_stage) >> 4);
                        const uint32_t zH = z_lo0 + ((zi * map.z_buf) >> 4) + q * ksteps * (4096u >> 4);
                        for (int jj = 0; jj < ksteps; ++jj) {
                            const uint32_t a = zH + jj * (4096u >> 4), b = xH + jj * ((2u * KD * 16u) >> 4);
                            tc_mma_f16_if(leader, dcol, pack64(a, kDescHi), pack64(b, kDescHi), IDESC_D, acc);
                            tc_mma_f16_if(leader, dcol, pack64(a, kDescHi), pack64(b + x_plane, kDescHi), IDESC_D, 1u);
                            tc_mma_f16_if(leader, dcol, pack64(a + z_plane, kDescHi), pack64(b, kDescHi), IDESC_D, 1u);
                            acc = 1;
                        }
                        tc_commit_if(leader, bar(BAR_X_EMPTY + st));
                        if (++st == xs) { st = 0; ph ^= 1u; }
                    }
                    if (!ok) break;
                    tc_commit_if(leader, bar(BAR_D_FULL + bank));
                    if (++bank == BANKS) { bank = 0; bank_ph ^= 1u; }
                }
            }
            if (!ok) break;
            tc_commit_if(leader, bar(BAR_Z_EMPTY + zi));
            if (++zi == zb) { zi = 0; z_ph ^= 1u; }
        }
        // every MMA issued by this thread must have completed before TMEM is freed
        tc_commit_if(leader, bar(BAR_MMA_DONE));
        mbar_wait_warp(bar(BAR_MMA_DONE), 0, abort_flag + 1, wl);
    } else {
        // ------------------------------------------------------------ MMA issuers: variance product, one warp per accumulator
        // The strips of all units go to the two accumulators in turn.  The two issuers share the k* chunks and run at their own
        // pace: while one's accumulator is being read back, the other's products keep the tensor cores busy.
        const uint32_t me = warp - 2, ring = ws / 2;
        const uint32_t w_lo0 = desc_addr(base + map.w + me * ring * (4u * KC * kStrip));
        const uint32_t wbar = me * (kMaxWS / 2);
        uint32_t w_s = 0, w_ph = 0, v_ph = 0;
        uint32_t t_base = 0, sigma = 0;      // chunks before the current pair, strips so far
        uint32_t zi = 0;                     // which group reads this unit's accumulators back
        bool ok = true;
        for (int unit = blockIdx.x; ok && unit < units; unit += unit_step, zi = zb == 2 ? zi ^ 1u : 0u) {
            const int part = part_of(unit);
            for (int p = prm.cut[part]; ok && p < prm.cut[part + 1]; ++p) {
                const Pair pr(p, S, nc);
                const uint32_t strips = pr.nb ? 2 : 1, which = (sigma & 1u) == me ? 0u : 1u;
                sigma += strips;
                if (which < strips) {
                    const int s = pr.a + which;
                    const uint32_t n_own = which ? pr.nb : pr.na, rows = (uint32_t)min(kStrip, nc * KC - s * kStrip);
                    if (!(ok = mbar_wait_warp(bar(BAR_V_EMPTY + me), v_ph ^ 1u, abort_flag, wl))) break;
                    for (uint32_t c = 0; c < n_own; ++c) {
                        const uint32_t t = t_base + c, slot = t % kSlots;
                        if (!(ok = mbar_wait_warp(bar(BAR_K_FULL + slot), (t / kSlots) & 1u, abort_flag, wl))) break;
                        if (!(ok = mbar_wait_warp(bar(BAR_W_FULL + wbar + w_s), w_ph, abort_flag, wl))) break;
                        tc_fence_after();
                        // In the strip's diagonal block the rows of W above the chunk's columns are zero (W is lower
                        // triangular): the MMAs start at the first row that can be non-zero and get narrower.
                        const uint32_t skip = (int)c > 4 * s ? (uint32_t)R3_IDX((c - 4 * s) * KC, rows, prm.status) : 0u;
                        const uint32_t idesc = instr_desc_f16(rows - skip);
                        const uint32_t vcol = tmem + me * kStrip + skip;
                        const uint32_t bH = (w_lo0 + (((uint32_t)R3_IDX(w_s, ring, prm.status) * (4u * KC * kStrip)) >> 4) + skip) | (rows << 16);
                        const uint32_t aK = tmem + kRingCol + slot * KC;
                        const uint32_t first = c > 0 ? 1u : 0u;
                        if (F8) {
                            // main term: FP16 hi x hi, two MMAs of depth 16; cross terms: one FP8 MMA of depth 32 each
                            // (planes after the FP16 hi plane: hi parts, then lo parts).  A slot holds, 8 columns each, the hi
                            // parts of the first 16 observations, all hi parts as E5M2, all lo parts as E5M2, the other 16 hi parts.
                            const uint32_t b8H = bH + ((rows * KC * 2u) >> 4), b8L = b8H + ((rows * KC) >> 4);
                            tc_mma_f16_ts_if(leader, vcol, aK, pack64(bH, kDescHi), idesc, first);
                            tc_mma_f16_ts_if(leader, vcol, aK + 24u, pack64(bH + 2u * rows, kDescHi), idesc, 1u);
                            // k* parts are E5M2; W's hi parts E4M3, its lo parts E5M2
                            tc_mma_f8_ts_if(leader, vcol, aK + 8u, pack64(b8L, kDescHi), instr_desc_f8(rows - skip, kFmtE5M2, kFmtE5M2), 1u);
                            tc_mma_f8_ts_if(leader, vcol, aK + 16u, pack64(b8H, kDescHi), instr_desc_f8(rows - skip, kFmtE5M2, kFmtE4M3), 1u);
                        } else {
                            // a slot holds, per 16 observations, 8 columns of hi parts and 8 of lo parts
                            const uint32_t bL = bH + ((rows * KC * 2u) >> 4);
#pragma unroll
                            for (int combo = 0; combo < 3; ++combo) {
                                const uint32_t a0 = combo == 2 ? aK + 8u : aK, b0 = combo == 1 ? bL : bH;
#pragma unroll
                                for (int jj = 0; jj < KC / 16; ++jj)
                                    tc_mma_f16_ts_if(leader, vcol, a0 + jj * 16u, pack64(b0 + jj * 2u * rows, kDescHi), idesc,
                                                     combo > 0 || jj > 0 ? 1u : first);
                            }
                        }
                        tc_commit_if(leader, bar(BAR_W_EMPTY + wbar + w_s));
                        if (++w_s == ring) { w_s = 0; w_ph ^= 1u; }
                        // slots go back to the distance products a bank at a time, when both issuers are through with it
                        if (t % KDC == KDC - 1) tc_commit_if(leader, bar(BAR_K_EMPTY + (t / KDC) % BANKS));
                    }
                    if (!ok) break;
                    tc_commit_if(leader, bar(BAR_V_FULL + 2 * me + zi));
                    v_ph ^= 1u;
                }
                // Chunks that only the other issuer takes (whole banks: strips have even numbers of chunks).  A wait by parity is
                // good for one phase, so this issuer waits for each of them too, and the bank is not free before it has: a slot
                // filled twice in between would look to it as if it had not been filled at all.
                for (uint32_t c = which < strips ? (which ? pr.nb : pr.na) : 0; ok && c < (uint32_t)pr.chunks(); ++c) {
                    const uint32_t t = t_base + c;
                    if (!(ok = mbar_wait_warp(bar(BAR_K_FULL + t % kSlots), (t / kSlots) & 1u, abort_flag, wl))) break;
                    if (t % KDC == KDC - 1 && leader) mbar_arrive(bar(BAR_K_EMPTY + (t / KDC) % BANKS));
                }
                t_base += pr.chunks();
            }
        }
        tc_commit_if(leader, bar(BAR_MMA_DONE + 1 + me));
        mbar_wait_warp(bar(BAR_MMA_DONE + 1 + me), 0, abort_flag + 1, wl);
    }
    } else if (warp < kFirstMatern) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIo));
        // ------------------------------------------------------------ candidates in, results out: a row per thread
        // Two buffers of scaled candidates: the candidates of the unit after the next come in once the present one's last strip
        // has been read back (its buffer is free when the Matern groups are through with it, and they are ahead of the products);
        // one buffer: those of the next unit, before that strip.  Two groups take every other unit each.
        const int io = (warp - kFirstIo) >> 2, row = (threadIdx.x - kFirstIo * 32) & (TILE_M - 1);
        const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        bool ok = true, bad = false;
        uint32_t z_ph = 0, v_ph = 0, red_ph = 0;     // parities per buffer b: bit b; v_ph: bit 2 b + accumulator
        uint32_t sigma = 0;                          // strips of all units so far
        float zn_in0 = 0.f, zn_in1 = 0.f;            // of the tiles in the buffers (the sign carries the out-of-range mark)
        const int groups = zb, own_step = unit_step * groups, ahead = unit_step * zb;   // a group per buffer
        auto strips_of = [&](int unit) { return min(S, 2 * prm.cut[part_of(unit) + 1]) - 2 * prm.cut[part_of(unit)]; };
        const int b = io;
        if (io < groups)
        for (int unit = (int)blockIdx.x + io * unit_step - ahead; ok && unit < units; unit += own_step) {
            const bool work = unit >= 0;
            const float zn_own = b ? zn_in1 : zn_in0;
            const int next = unit + ahead;
            const int part = work ? part_of(unit) : 0;
            const int s0 = work ? 2 * prm.cut[part] : 0, s1 = work ? s0 + strips_of(unit) : 0;
            const int at = !work ? -1 : zb == 1 ? s1 - 1 : s1;
            if (groups == 2 && unit >= unit_step) sigma += strips_of(unit - unit_step);   // the other group's
            double q_acc = 0.0;
            for (int s = work ? s0 : -1; s <= s1; ++s) {
                if (s == at && next < units) {
                    // ---- scale a candidate, split it, store it as the A operand of the distance product
                    ok = mbar_wait_warp(bar(BAR_Z_EMPTY + b), ((z_ph >> b) & 1u) ^ 1u, abort_flag, wl);
                    if (!ok) break;
                    const uint32_t tile = tile_of(next);
                    const int g = (int)(tile / tiles_per_gp);
                    const long long cand = (long long)(tile - g * tiles_per_gp) * TILE_M + row;
                    const bool valid = cand < prm.m;
                    float zn = 0.f;
                    bool far = false;
                    const float* zrow =
                        prm.xcand + (size_t)R3_IDX((long long)g * prm.m + (valid ? cand : 0), (long long)prm.batch * prm.m, prm.status) * prm.d;
                    if (next + unit_step < units) {   // the row after that: on its way to L2
                        const uint32_t nt = tile_of(next + unit_step), ng = nt / tiles_per_gp;
                        const long long nr = (long long)(nt - ng * tiles_per_gp) * TILE_M + row;
                        if (nr < prm.m) {
                            const char* pf = reinterpret_cast<const char*>(prm.xcand + ((size_t)ng * prm.m + nr) * prm.d);
                            for (int off = 0; off < prm.d * 4; off += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf + off));
                        }
                    }
                    const float* cen = prm.centre + (size_t)g * DP;
                    const float* scl = prm.scale + (size_t)g * DP;
                    const bool vec = (prm.d % 4) == 0 && (reinterpret_cast<uintptr_t>(prm.xcand) & 15) == 0;
                    uint8_t* zdst = sm + map.z + b * map.z_buf + row * 16;
                    auto load4 = [&](int j4) {
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (vec && 4 * j4 < prm.d) {
                            // read once: streaming load, so that the pool does not push W out of L2
                            v = __ldcs(reinterpret_cast<const float4*>(zrow + 4 * j4));
                        } else if (4 * j4 < prm.d) {
                            v.x = __ldcs(zrow + 4 * j4);
                            v.y = (4 * j4 + 1 < prm.d) ? __ldcs(zrow + 4 * j4 + 1) : 0.f;
                            v.z = (4 * j4 + 2 < prm.d) ? __ldcs(zrow + 4 * j4 + 2) : 0.f;
                            v.w = (4 * j4 + 3 < prm.d) ? __ldcs(zrow + 4 * j4 + 3) : 0.f;
                        }
                        return v;
                    };
                    // 8 features per step; the next step's loads are under way while this one is scaled and split.  (The loop is kept
                    // short on purpose, as all code of this kernel is: see the top of the file.)
                    float4 nxt[2] = {load4(0), load4(1)};
#pragma unroll 1
                    for (int j8 = 0; j8 < DP / 8; ++j8) {
                        const float4 cur[2] = {nxt[0], nxt[1]};
                        nxt[0] = load4(2 * j8 + 2);
                        nxt[1] = load4(2 * j8 + 3);
                        __half2 hi[4], lo[4];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int j4 = 2 * j8 + h;
                            const float z[4] = {cur[h].x, cur[h].y, cur[h].z, cur[h].w};
                            const float4 c4 = __ldg(reinterpret_cast<const float4*>(cen + R3_IDX(4 * j4, DP - 3, prm.status)));
                            const float4 s4 = __ldg(reinterpret_cast<const float4*>(scl + R3_IDX(4 * j4, DP - 3, prm.status)));
                            const float cc[4] = {c4.x, c4.y, c4.z, c4.w}, ss[4] = {s4.x, s4.y, s4.z, s4.w};
                            float zt[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                bad |= !isfinite(z[e]);
                                float v = valid ? (z[e] - cc[e]) * ss[e] : 0.f;
                                if (fabsf(v) > kMaxScaled) {   // outside the FP16 planes' range: clamp, and have it recomputed
                                    v = copysignf(kMaxScaled, v);
                                    far = true;
                                }
                                zt[e] = v;
                                zn = fmaf(v, v, zn);
                            }
                            split2(zt[0], zt[1], hi[2 * h], lo[2 * h]);
                            split2(zt[2], zt[3], hi[2 * h + 1], lo[2 * h + 1]);
                            if (Z32)
                                *reinterpret_cast<float4*>(sm + map.z32 + b * map.z32_buf + (j4 * TILE_M + row) * 16) =
                                    make_float4(zt[0], zt[1], zt[2], zt[3]);
                        }
                        *reinterpret_cast<uint4*>(zdst + j8 * 2048u) = *reinterpret_cast<const uint4*>(hi);
                        *reinterpret_cast<uint4*>(zdst + 256u * DP + j8 * 2048u) = *reinterpret_cast<const uint4*>(lo);
                    }
                    float* znb = zn_buf(b);
                    const float kvscale = prm.kscale[g] * prm.sf2[g];   // k* = sf2 * (k*/sf2), scaled for its FP16 split
                    znb[row] = zn;
                    znb[TILE_M + row] = far ? INFINITY : kvscale * kRefine / (zn + prm.xnmax[g]);
                    if (row == 0) *reinterpret_cast<float4*>(znb + 2 * TILE_M) = make_float4(kvscale, 1.f / prm.kscale[g], __int_as_float(g), 0.f);
                    zn = far ? -zn : zn;
                    if (b) zn_in1 = zn;
                    else zn_in0 = zn;
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(BAR_Z_FULL + b));
                    z_ph ^= 1u << b;
                }
                if (!work || s == s1) break;
                // ---- a finished strip: q += sum_i V^2, then the accumulator is free
                const uint32_t v_s = sigma++ & 1u;
                ok = mbar_wait(bar(BAR_V_FULL + 2 * v_s + b), (v_ph >> (2 * b + v_s)) & 1u, abort_flag, wl);
                v_ph ^= 1u << (2 * b + v_s);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                const int rows = min(kStrip, nc * KC - s * kStrip);
#pragma unroll 1
                for (int c0 = 0; c0 < rows; c0 += 32) {   // two column blocks per round trip to tensor memory
                    float v[16], w[16];
                    tc_ld16_issue(lane_addr + v_s * kStrip + c0, v);
                    tc_ld16_issue(lane_addr + v_s * kStrip + c0 + 16, w);
                    tc_wait_ld32(v, w);
                    uint64_t part0 = 0, part1 = 0;
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const uint64_t v2 = pack2(v[i], v[i + 1]), w2 = pack2(w[i], w[i + 1]);
                        part0 = fma2(v2, v2, part0);
                        part1 = fma2(w2, w2, part1);
                    }
                    float a0, a1, b0, b1;
                    unpack2(part0, a0, a1);
                    unpack2(part1, b0, b1);
                    q_acc += (double)(a0 + a1);
                    q_acc += (double)(b0 + b1);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(BAR_V_EMPTY + v_s));
            }
            if (!ok) break;
            if (!work) continue;
            // ---- the groups' partial sums; a tile whose pairs went to several units is finished by the last of them, each 32
            // rows by the warp that sees its last part arrive
            ok = mbar_wait_warp(bar(BAR_RED_FULL + b), (red_ph >> b) & 1u, abort_flag, wl);
            if (!ok) break;
            double mu_acc = 0.0, a2_acc = 0.0, s2_acc = 0.0;
#pragma unroll
            for (int gg = 0; gg < G; ++gg) {
                const double* o = reinterpret_cast<const double*>(sm + map.red + b * map.red_buf) + gg * (3 * TILE_M) + row;
                mu_acc += o[0];
                a2_acc += o[TILE_M];
                s2_acc += o[2 * TILE_M];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_RED_EMPTY + b));
            red_ph ^= 1u << b;
            const uint32_t tile = tile_of(unit);
            bool finish = true;
            if (prm.splits > 1) {
                const size_t slot = (size_t)(unit % tiles) * prm.splits;
                double* mine = prm.partial + (slot + part) * (4 * TILE_M) + row;
                __stcg(mine, mu_acc);
                __stcg(mine + TILE_M, q_acc);
                __stcg(mine + 2 * TILE_M, a2_acc);
                __stcg(mine + 3 * TILE_M, s2_acc);
                __threadfence();
                __syncwarp();
                int before = 0;   // parts of these 32 rows that are already there
                if (lane == 0) before = atomicAdd(prm.arrived + R3_IDX((unit % tiles) * 4 + (warp & 3), tiles * 4, prm.status), 1);
                finish = __shfl_sync(0xffffffffu, before, 0) == prm.splits - 1;
                if (finish) {
                    __threadfence();
                    mu_acc = q_acc = a2_acc = s2_acc = 0.0;
#pragma unroll 1
                    for (int i = 0; i < prm.splits; ++i) {
                        const double* o = prm.partial + (slot + i) * (4 * TILE_M) + row;
                        mu_acc += __ldcg(o);
                        q_acc += __ldcg(o + TILE_M);
                        a2_acc += __ldcg(o + 2 * TILE_M);
                        s2_acc += __ldcg(o + 3 * TILE_M);
                    }
                }
            }
            const int g = (int)(tile / tiles_per_gp);
            const long long cand = (long long)(tile - g * tiles_per_gp) * TILE_M + row;
            float ei_mine = 0.f;
            if (finish && cand < prm.m) {
                const bool far_cand = zn_own < 0.f;
                q_acc *= prm.vinv2[g];   // undo the power-of-two scaling of k* and W
                const size_t f = (size_t)R3_IDX((long long)g * prm.m + cand, (long long)prm.batch * prm.m, prm.status);
                const CandidateResult res =
                    finalize_candidate(mu_acc, q_acc, (double)prm.sf2[g], (double)prm.best[R3_IDX(g, prm.batch, prm.status)]);
                __stcs(prm.mu + f, res.mu);
                __stcs(prm.sigma + f, res.sigma);
                __stcs(prm.ei + f, res.ei);
                if (res.ei == res.ei) ei_mine = res.ei;
                const double eps = far_cand ? 1.0 : kEpsTc0 + kEpsTc1 * prm.rsqrt_dp * (double)(fabsf(zn_own) + prm.xnmax[g]);
                prm.err_mu[f] = mu_error_estimate(eps, a2_acc);
                prm.err_q[f] = q_error_estimate(F8 && !far_cand ? eps + kEpsF8 : eps, prm.wnorm[g], q_acc, s2_acc);
            }
            if (finish) {   // EI >= 0: the order of the bits is the order of the values
                const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(ei_mine));
                if (lane == 0)
                    prm.tile_max[R3_IDX((long long)tile * 4 + (warp & 3), 4ll * tiles_per_gp * prm.batch, prm.status)] = __uint_as_float(top);
            }
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(prm.status, DEV_NONFINITE);
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsMatern));
        // ------------------------------------------------------------ Matern warp groups
        const int grp = (warp - kFirstMatern) >> 2;   // 0..G-1
        const int row = ((warp & 3) << 5) + lane;   // candidate row in the tile == TMEM lane
        const uint32_t ring_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + kRingCol;
        uint32_t t = grp, t_base = 0;            // next own chunk, and the chunks before the current pair (all units' numbering)
        int zi = 0;
        uint32_t z_ph = 0, tile_iter = 0;
        bool ok = true;
        for (int unit = blockIdx.x; ok && unit < units; unit += unit_step, ++tile_iter) {
            const int part = part_of(unit);
            ok = mbar_wait_warp(bar(BAR_Z_FULL + zi), z_ph, abort_flag, wl);
            if (!ok) break;
            const float* znb = zn_buf(zi);
            const float zn = znb[row], v_thresh = znb[TILE_M + row];
            const float4 tile_s = *reinterpret_cast<const float4*>(znb + 2 * TILE_M);
            const float kvscale = tile_s.x, inv = tile_s.y;   // inv: scaled k* -> k*, a power of two
            const int g = __float_as_int(tile_s.z);
            const int quads = prm.d <= 8 ? (prm.d + 3) / 4 : 4;   // FEW: groups of four features (three are no faster than four)
            const uint64_t zn2 = pack2(zn, zn), minus2 = pack2(-2.f, -2.f);
            const uint64_t pc0 = pack2(kvscale, kvscale), pc1 = pack2(kvscale * kPolyC1, kvscale * kPolyC1),
                           pc2 = pack2(kvscale * kPolyC2, kvscale * kPolyC2);
            const float* xs_g = prm.xs32 + (size_t)g * prm.NP * DP;
            const float* xn_g = prm.xnorm + (size_t)g * prm.NP;
            const float* al_g = prm.alpha + (size_t)g * prm.NP;
            double mu_acc = 0.0, a2_acc = 0.0, s2_acc = 0.0;   // the last two: scales of the error estimate
            for (int p = prm.cut[part]; ok && p < prm.cut[part + 1]; ++p) {
                const uint32_t chunks = (uint32_t)Pair(p, S, nc).chunks();
                for (; ok && t - t_base < chunks; t += G) {
                    const int c = (int)(t - t_base);
                    const uint32_t u = t / KDC;
                    ok = mbar_wait_warp(bar(BAR_D_FULL + u % BANKS), (u / BANKS) & 1u, abort_flag, wl);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t slot_addr = ring_addr + (t % kSlots) * KC;
                    float dots[F8 ? 2 : 1][16];
                    if (F8) {   // the 8-bit planes of both halves lie over the second half's dot products
                        tc_ld16_issue(slot_addr, dots[0]);
                        tc_ld16_issue(slot_addr + 16, dots[F8]);
                        tc_wait_ld32(dots[0], dots[F8]);
                    }
                    const bool fresh = c >= 8 * p;   // first time this chunk is generated for the tile
                    uint32_t f8h[2][4], f8l[2][4];
                    constexpr int kUnroll = F8 ? 2 : 1;   // one copy of the loop's body where registers allow it: see above
#pragma unroll kUnroll
                    for (int h = 0; h < 2; ++h) {
                        if (!F8) tc_ld16_issue(slot_addr + h * 16, dots[0]);
                        const float* dot16 = dots[F8 ? h : 0];
                        const int k0 = (int)R3_IDX(c * KC + h * 16, prm.NP - 15, prm.status);
                        ulonglong2 xn[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) xn[q] = __ldg(reinterpret_cast<const ulonglong2*>(xn_g + k0 + 4 * q));
                        if (!F8) tc_wait_ld16(dots[0]);
                        uint64_t v2[8];   // k* times kvscale (the power of two of its FP16 split), in pairs
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            float r0, r1;
                            unpack2(fma2(minus2, pack2(dot16[2 * e], dot16[2 * e + 1]), add2(zn2, e & 1 ? xn[e / 2].y : xn[e / 2].x)), r0, r1);
                            // |.|: a slightly negative r^2 (rounding) is a tiny distance either way
                            const float u0 = sqrt_approx(fabsf(r0)), u1 = sqrt_approx(fabsf(r1));
                            const uint64_t uu = pack2(u0, u1);
                            v2[e] = mul2(fma2(uu, fma2(uu, pc2, pc1), pc0), pack2(exp2_approx(-u0), exp2_approx(-u1)));
                        }
                        // largest of the sixteen in eight three-input maxima
                        float m8[8];
#pragma unroll
                        for (int e = 0; e < 8; e += 2) {
                            float a0, a1, b0, b1;
                            unpack2(v2[e], a0, a1);
                            unpack2(v2[e + 1], b0, b1);
                            m8[e / 2] = max3(a0, a1, b0);
                            m8[4 + e / 2] = b1;
                        }
                        const float vmax = max3(max3(m8[0], m8[1], m8[2]), max3(m8[3], m8[4], m8[5]), max3(m8[6], m8[7], 0.f));
                        if (vmax > v_thresh) {   // close pairs of this candidate
                            float kv[16];
                            uint32_t marked = 0;
#pragma unroll
                            for (int e = 0; e < 8; ++e) unpack2(v2[e], kv[2 * e], kv[2 * e + 1]);
                            if (Z32) {   // direct differences, inline
#pragma unroll
                                for (int i = 0; i < 16; ++i) marked |= (kv[i] > v_thresh) ? (1u << i) : 0u;
                                const float4* zr = reinterpret_cast<const float4*>(sm + map.z32 + zi * map.z32_buf + row * 16);
                                for (; marked; marked &= marked - 1) {
                                    const uint32_t i = (uint32_t)__ffs(marked) - 1u;
                                    const float4* xp = reinterpret_cast<const float4*>(xs_g + (size_t)(k0 + (int)i) * DP);
                                    float acc0 = 0.f, acc1 = 0.f;
#pragma unroll 4
                                    for (int e = 0; e < (FEW ? quads : DP / 4); ++e) {
                                        const float4 x4 = __ldg(xp + e), z4 = zr[e * TILE_M];
                                        float df = z4.x - x4.x;
                                        acc0 = fmaf(df, df, acc0);
                                        df = z4.y - x4.y;
                                        acc1 = fmaf(df, df, acc1);
                                        df = z4.z - x4.z;
                                        acc0 = fmaf(df, df, acc0);
                                        df = z4.w - x4.w;
                                        acc1 = fmaf(df, df, acc1);
                                    }
                                    const float uu = sqrtf(acc0 + acc1);
                                    const float val = kvscale * fmaf(uu, fmaf(uu, kPolyC2, kPolyC1), 1.f) * exp2f(-uu);
                                    if constexpr (FEW) {
                                        kv[i] = val;
                                    } else {
#pragma unroll
                                        for (int e2 = 0; e2 < 16; ++e2) kv[e2] = (uint32_t)e2 == i ? val : kv[e2];
                                    }
                                }
                            } else {
                                // rare: out of line, through a local array; values refined in an earlier pair of strips come back
                                // from the tile's cache
                                const uint32_t key0 = ((tile_iter & 0x3ffffu) << 13) | (uint32_t)k0;
                                unsigned long long* slots = reinterpret_cast<unsigned long long*>(sm + map.cache) + row * kCacheSlots;
                                refine_close_pairs_smem(kv, v_thresh, kvscale, sm + map.z + zi * map.z_buf + row * 16, DP,
                                                        xs_g + (size_t)k0 * DP, S > 2 ? slots : nullptr, key0, !fresh);
                            }
#pragma unroll
                            for (int e = 0; e < 8; ++e) v2[e] = pack2(kv[2 * e], kv[2 * e + 1]);
                        }
                        __syncwarp();   // the stores to tensor memory are warp-wide
                        if (fresh) {   // warp-uniform: the mean and the error scales see every observation once
                            uint64_t mp = 0, ap = 0, sp = 0;
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const ulonglong2 al = __ldg(reinterpret_cast<const ulonglong2*>(al_g + k0 + 4 * q));
#pragma unroll
                                for (int e = 0; e < 2; ++e) {
                                    const uint64_t v = v2[2 * q + e], va = mul2(v, e ? al.y : al.x);
                                    mp = add2(mp, va);
                                    ap = fma2(va, va, ap);
                                    sp = fma2(v, v, sp);
                                }
                            }
                            float m0, m1, a0, a1, b0, b1;
                            unpack2(mp, m0, m1);
                            unpack2(ap, a0, a1);
                            unpack2(sp, b0, b1);
                            mu_acc += (double)(m0 + m1);
                            a2_acc += (double)(a0 + a1);
                            s2_acc += (double)(b0 + b1);
                        }
                        // split into the FP16 planes and over the dot products they came from
                        uint32_t out[16];
                        if (F8) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                float v4[4];
                                unpack2(v2[2 * e], v4[0], v4[1]);
                                unpack2(v2[2 * e + 1], v4[2], v4[3]);
                                split4_f8(v4, out[2 * e], out[2 * e + 1], f8h[h][e], f8l[h][e]);
                            }
                            tc_st8(slot_addr + (h ? 24 : 0), out);
                        } else {
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                float a, b;
                                unpack2(v2[e], a, b);
                                const __half2 hi = __floats2half2_rn(a, b);
                                const __half2 lo = __floats2half2_rn(minus_half(a, __low2half(hi)), minus_half(b, __high2half(hi)));
                                out[e] = *reinterpret_cast<const uint32_t*>(&hi);
                                out[8 + e] = *reinterpret_cast<const uint32_t*>(&lo);
                            }
                            tc_st16(slot_addr + h * 16, out);
                        }
                    }
                    if (F8) {
                        uint32_t o8[16];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            o8[e] = f8h[0][e];
                            o8[4 + e] = f8h[1][e];
                            o8[8 + e] = f8l[0][e];
                            o8[12 + e] = f8l[1][e];
                        }
                        tc_st16(slot_addr + 8, o8);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(BAR_K_FULL + t % kSlots));
                }
                t_base += chunks;
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_Z_EMPTY + zi));
            ok = mbar_wait_warp(bar(BAR_RED_EMPTY + zi), z_ph ^ 1u, abort_flag, wl);
            if (!ok) break;
            double* o = reinterpret_cast<double*>(sm + map.red + zi * map.red_buf) + R3_IDX(grp * (3 * TILE_M) + row, G * 3 * TILE_M, prm.status);
            const double inv64 = (double)inv, inv2 = inv64 * inv64;
            o[0] = mu_acc * inv64;
            o[TILE_M] = a2_acc * inv2;
            o[2 * TILE_M] = s2_acc * inv2;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_RED_FULL + zi));
            if (++zi == zb) { zi = 0; z_ph ^= 1u; }
        }
    }

    // ---------------------------------------------------------------- teardown
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomicOr(prm.status, DEV_TIMEOUT);
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------
// operand preparation (fit time)
__global__ void centre_kernel(const float* __restrict__ X, const float* __restrict__ inv_ell, int n, int d, int DP,
                              float* __restrict__ centre, float* __restrict__ scale)
{
    __shared__ double s[256];
    const int g = blockIdx.y, j = blockIdx.x;
    double acc = 0.0;
    if (j < d)
        for (int i = threadIdx.x; i < n; i += 256) acc += (double)X[((size_t)g * n + i) * d + j];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        centre[(size_t)g * DP + j] = (j < d) ? (float)(s[0] / n) : 0.f;
        scale[(size_t)g * DP + j] = (j < d) ? (float)((double)inv_ell[(size_t)g * d + j] * kCoordScale) : 0.f;
    }
}

// One block per (distance product, GP): scaled observations as FP16 hi/lo planes in the MMA's
// B-operand layout, their squared norms (of the FP32 values the planes represent), the padded weights,
// and the largest scaled coordinate (the FP16 planes have a limited range).
__global__ void xt_build_kernel(const float* __restrict__ X, const float* __restrict__ centre,
                                const float* __restrict__ scale, const float* __restrict__ alpha32, int n, int d,
                                int npad_fit, int DP, int parts, int NP, int KD, __half* __restrict__ xt,
                                float* __restrict__ xs32, float* __restrict__ xnorm, float* __restrict__ alpha, unsigned* __restrict__ xamax_bits,
                                unsigned* __restrict__ xnmax_bits)
{
    const int g = blockIdx.y, c = blockIdx.x;
    float nmax = 0.f;
    __half* blob = xt + ((size_t)g * (NP / KD) + c) * (2 * DP * KD);
    const float* cen = centre + (size_t)g * DP;
    const float* scl = scale + (size_t)g * DP;
    float amax = 0.f;
    for (int e = threadIdx.x; e < DP * KD; e += blockDim.x) {
        const int r = e % KD, j = e / KD;
        const int k = c * KD + r;
        float xv = 0.f;
        if (k < n && j < d) xv = (float)(((double)X[((size_t)g * n + k) * d + j] - (double)cen[j]) * (double)scl[j]);
        amax = fmaxf(amax, fabsf(xv));
        xs32[((size_t)g * NP + k) * DP + j] = xv;
        const __half h = __float2half_rn(xv);
        const int DPp = DP / parts, jp = j % DPp;
        const size_t off = (size_t)(j / DPp) * (2 * DPp * KD) + ((size_t)(jp / 8) * KD + r) * 8 + (jp % 8);
        blob[off] = h;
        blob[(size_t)DPp * KD + off] = __float2half_rn(xv - __half2float(h));
    }
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if ((threadIdx.x & 31) == 0) atomicMax(xamax_bits, __float_as_uint(amax));
    for (int r = threadIdx.x; r < KD; r += blockDim.x) {
        const int k = c * KD + r;
        double nrm = 0.0;
        if (k < n)
            for (int j = 0; j < d; ++j) {
                const float xv = (float)(((double)X[((size_t)g * n + k) * d + j] - (double)cen[j]) * (double)scl[j]);
                nrm += (double)xv * (double)xv;
            }
        xnorm[(size_t)g * NP + k] = (float)nrm;
        nmax = fmaxf(nmax, (float)nrm);
        alpha[(size_t)g * NP + k] = (k < n) ? alpha32[(size_t)g * npad_fit + k] : 0.f;
    }
    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(nmax));   // order-preserving for nmax >= 0
    if ((threadIdx.x & 31) == 0) atomicMax(xnmax_bits + g, top);
}

// Powers of two that the operands of the variance product are multiplied by: 2^sw W and 2^sk k*.
__host__ __device__ inline void operand_scales(float wmax, float sf2, bool f8, int& sw, int& sk)
{
    int ew = 0, ek = 0;
    frexp((double)wmax, &ew);   // wmax < 2^ew
    frexp((double)sf2, &ek);    // sf2  < 2^ek  (k* <= sf2)
    sw = (f8 ? kScaleExpF8 : kScaleExp) - ew;
    sk = kScaleExp - ek;
}

// One block per (chunk c, strip s, GP): the block of 2^eW W (rows 128 s.., columns c KC..) as FP16 hi/lo planes in the
// B-operand layout; zero outside the lower triangle and outside n.  A thread takes eight consecutive columns of a row: it
// reads 64 contiguous bytes and writes 16 to each plane.
// With f8 the second plane holds, instead of the FP16 lo parts, two 8-bit planes in the 8-bit form of the same
// layout (16 k-elements per 16-byte slice): the hi parts as E4M3 (|2^eW W| < 2^8 for these histories), then the
// lo parts as E5M2.  strip_rows: 128, or 256 for the paired kernel's passes.
__global__ void wt_build_kernel(const double* __restrict__ W64, int n, int npad_fit, int strip_rows, int nc, size_t gp_stride,
                                const unsigned* __restrict__ wmax, const float* __restrict__ sf2, float* __restrict__ kscale,
                                double* __restrict__ vinv2, __half* __restrict__ wt, bool f8)
{
    const int c = blockIdx.x, s = blockIdx.y, g = blockIdx.z, per = strip_rows / KC;
    if (c >= (s + 1) * per) return;
    const int rows = min(strip_rows, nc * KC - s * strip_rows);
    __half* dst = wt + (size_t)g * gp_stride + (size_t)per * s * (s + 1) / 2 * (2 * KC * strip_rows) + (size_t)c * (2 * KC * rows);
    const double* Wg = W64 + (size_t)g * npad_fit * npad_fit;
    int sw, sk;
    operand_scales(__uint_as_float(wmax[g]), sf2[g], f8, sw, sk);
    const double sc = ldexp(1.0, sw);
    if (c == 0 && s == 0 && threadIdx.x == 0) {
        kscale[g] = (float)ldexp(1.0, sk);
        vinv2[g] = ldexp(1.0, -2 * (sw + sk));
    }
    for (int e = threadIdx.x; e < rows * (KC / 8); e += blockDim.x) {
        const int k8 = e % (KC / 8), r = e / (KC / 8);
        const int i = s * strip_rows + r, k = c * KC + k8 * 8;
        float w[8] = {};
        if (i < n && k <= i) {   // a row of W has npad_fit >= i + 1 columns, a multiple of 32
            const double2* src = reinterpret_cast<const double2*>(Wg + (size_t)i * npad_fit + k);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const double2 v = src[q];
                w[2 * q] = k + 2 * q <= i ? (float)(v.x * sc) : 0.f;
                w[2 * q + 1] = k + 2 * q + 1 <= i ? (float)(v.y * sc) : 0.f;
            }
        }
        __half2 hi[4];
        float lo[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            hi[q] = __floats2half2_rn(w[2 * q], w[2 * q + 1]);
            const float2 back = __half22float2(hi[q]);
            lo[2 * q] = w[2 * q] - back.x;
            lo[2 * q + 1] = w[2 * q + 1] - back.y;
            w[2 * q] = back.x;
            w[2 * q + 1] = back.y;
        }
        const size_t off = ((size_t)k8 * rows + r) * 8;
        *reinterpret_cast<uint4*>(dst + off) = *reinterpret_cast<const uint4*>(hi);
        if (f8) {
            uint8_t* d8 = reinterpret_cast<uint8_t*>(dst + (size_t)KC * rows);
            const size_t off8 = ((size_t)(k8 / 2) * rows + r) * 16 + (k8 % 2) * 8;
            *reinterpret_cast<uint2*>(d8 + off8) = make_uint2(e4m3x4(w[0], w[1], w[2], w[3]), e4m3x4(w[4], w[5], w[6], w[7]));
            *reinterpret_cast<uint2*>(d8 + (size_t)KC * rows + off8) =
                make_uint2(e5m2x4(lo[0], lo[1], lo[2], lo[3]), e5m2x4(lo[4], lo[5], lo[6], lo[7]));
        } else {
            __half2 l2[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) l2[q] = __floats2half2_rn(lo[2 * q], lo[2 * q + 1]);
            *reinterpret_cast<uint4*>(dst + (size_t)KC * rows + off) = *reinterpret_cast<const uint4*>(l2);
        }
    }
}

TensorOperands* ops_of(const r3_fit_state* gp) { return static_cast<TensorOperands*>(gp->tc); }

constexpr int kF8MinPasses = 8;   // pairs of strips (n > 1792): below that the guard hands more candidates to the FP64 pass than the cheaper MMAs save

// The kernel a set of operands runs on, with or without FP8 cross terms
void (*kernel_of(const TensorOperands* t, bool f8))(const TcParams)
{
    const bool z32 = t->DP <= kZ32MaxDP, few = t->DP <= 16;
    if (f8) return few ? score_tc_kernel<true, true, true> : z32 ? score_tc_kernel<true, true, false> : score_tc_kernel<true, false, false>;
    return few ? score_tc_kernel<false, true, true> : z32 ? score_tc_kernel<false, true, false> : score_tc_kernel<false, false, false>;
}

int env_int(const char* name, int fallback)
{
    const char* v = getenv(name);
    return v ? atoi(v) : fallback;
}

}  // namespace

bool tc_supported(int n, int d) { return n >= 1 && n <= kMaxN && d >= 1 && d <= 128; }

void tc_release(r3_fit_state& st)
{
    TensorOperands* t = ops_of(&st);
    if (!t) return;
    dev_free(t->centre);
    dev_free(t->scale);
    dev_free(t->xt);
    dev_free(t->xs32);
    dev_free(t->xnorm);
    dev_free(t->alpha);
    dev_free(t->wt);
    dev_free(t->kscale);
    dev_free(t->vinv2);
    dev_free(t->wt16);
    dev_free(t->vinv2_16);
    delete t;
    st.tc = nullptr;
}

r3_status_t tc_prepare(r3_fit_state& st, int device, cudaStream_t stream)
{
    const int B = st.batch, n = st.n, d = st.d;
    TensorOperands* t = new (std::nothrow) TensorOperands;
    if (!t) {
        set_error("out of host memory");
        return R3_ERR_ALLOC;
    }
    st.tc = t;
    // R3_TC_PAIR=1 lays the operands out for the paired kernel (r3_score_tc2.cu) where that serves the shape
    const int want_f8 = env_int("R3_TC_F8", -1);
    t->f8 = want_f8 >= 0 ? want_f8 != 0 && n > 128 : (n + 255) / 256 >= kF8MinPasses;
    t->DP = round_up(d, 16);
    t->KD = KD;
    t->NP = round_up(n, 256);
    t->P = t->NP / 256;
    int pair_ws = 0;
    t->pair = env_int("R3_TC_PAIR", 0) != 0 && !t->f8 && tc_pair_fits(t, &pair_ws);
    if (!t->pair) {
        t->parts = (t->DP + kPartDP - 1) / kPartDP;
        t->DP = t->parts * round_up((t->DP + t->parts - 1) / t->parts, 16);
        t->NP = round_up(n, KD);
        t->S = (n + kStrip - 1) / kStrip;
        t->P = (t->S + 1) / 2;
        t->G = G;
        const size_t budget = 227 * 1024 - 1024;
        t->zb = 2;
        t->xs = 2;
        t->ws = 6;   // four per accumulator instead of three: no faster (512 observations) or slower (701 by 0.1 ms in 0.6)
        auto bytes = [&] { return (size_t)smem_map(t->DP, t->parts, t->zb, t->xs, t->ws).end; };
        if (bytes() > budget) t->zb = 1;
        while (t->ws > 4 && bytes() > budget) t->ws -= 2;
        if (bytes() > budget) {
            tc_release(st);   // does not fit: the SIMT engine serves this shape
            return R3_OK;
        }
        t->smem_bytes = bytes() + 1024;
    }
    const int strip_rows = t->pair ? 256 : kStrip, strips = t->pair ? t->P : t->S, chunks = t->NP / KC, per = strip_rows / KC;
    const int last_rows = t->NP - (strips - 1) * strip_rows;
    t->wt_gp_stride = (size_t)per * strips * (strips - 1) / 2 * (2 * KC * strip_rows) + (size_t)chunks * (2 * KC * last_rows);
    auto fail = [&](const char* what, cudaError_t e) {
        set_error("%s failed: %s", what, cudaGetErrorString(e));
        cudaStreamSynchronize(stream);
        FreeScope no_wait;
        tc_release(st);
        return e == cudaErrorMemoryAllocation ? R3_ERR_ALLOC : R3_ERR_CUDA;
    };
    cudaError_t e;
    if ((e = dev_malloc(&t->centre, sizeof(float) * B * t->DP)) != cudaSuccess) return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->scale, sizeof(float) * B * t->DP)) != cudaSuccess) return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->xt, sizeof(__half) * B * (size_t)(t->NP / t->KD) * 2 * t->DP * t->KD)) != cudaSuccess)
        return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->xs32, sizeof(float) * B * (size_t)t->NP * t->DP)) != cudaSuccess) return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->xnorm, sizeof(float) * B * t->NP)) != cudaSuccess) return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->alpha, sizeof(float) * B * t->NP)) != cudaSuccess) return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->wt, sizeof(__half) * B * t->wt_gp_stride)) != cudaSuccess) return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->kscale, sizeof(float) * B)) != cudaSuccess) return fail("cudaMalloc", e);
    if ((e = dev_malloc(&t->vinv2, sizeof(double) * B)) != cudaSuccess) return fail("cudaMalloc", e);
    if (t->f8 && (dev_malloc(&t->wt16, sizeof(__half) * B * t->wt_gp_stride) != cudaSuccess ||
                  dev_malloc(&t->vinv2_16, sizeof(double) * B) != cudaSuccess)) {
        cudaGetLastError();   // no memory for the second form: every pool is scored with FP8 cross terms
        FreeScope no_wait;    // nothing has used them yet
        dev_free(t->wt16);
        dev_free(t->vinv2_16);
        t->wt16 = nullptr;
        t->vinv2_16 = nullptr;
    }
    t->xnmax = reinterpret_cast<float*>(st.xnmax_d);   // lives in the state's block

    // scaled observations (their largest coordinate decides whether the FP16 planes can hold them), then the planes of W,
    // scaled by a power of two that the largest |W| decides
    centre_kernel<<<dim3(t->DP, B), 256, 0, stream>>>(st.X, st.inv_ell, n, d, t->DP, t->centre, t->scale);
    xt_build_kernel<<<dim3(t->NP / t->KD, B), 256, 0, stream>>>(st.X, t->centre, t->scale, st.alpha32, n, d, st.npad, t->DP,
                                                                t->parts, t->NP, t->KD, t->xt, t->xs32, t->xnorm, t->alpha, st.xamax_d,
                                                                st.xnmax_d);
    wt_build_kernel<<<dim3(chunks, strips, B), 256, 0, stream>>>(st.W64, n, st.npad, strip_rows, chunks, t->wt_gp_stride, st.wmax_d,
                                                                 st.sf2_d, t->kscale, t->vinv2, t->wt, t->f8);
    g_launches += 3;
    if (t->wt16) {
        wt_build_kernel<<<dim3(chunks, strips, B), 256, 0, stream>>>(st.W64, n, st.npad, strip_rows, chunks, t->wt_gp_stride,
                                                                     st.wmax_d, st.sf2_d, t->kscale, t->vinv2_16, t->wt16, false);
        ++g_launches;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return fail("operand preparation launch", e);
    if (t->pair) return R3_OK;
    // The cap on dynamic shared memory belongs to the kernel, not to the handle, and handles with different
    // feature counts share an instantiation with different sizes: raise it to the device's limit (the kernel
    // has no static shared memory), so that no handle's preparation lowers it for another.
    int smem_optin = 0;
    if ((e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device)) != cudaSuccess)
        return fail("cudaDeviceGetAttribute", e);
    if ((size_t)smem_optin < t->smem_bytes) {
        cudaStreamSynchronize(stream);
        FreeScope no_wait;
        tc_release(st);   // the SIMT engine serves this history
        return R3_OK;
    }
    for (int form = 0; form < (t->f8 ? 2 : 1); ++form) {
        e = cudaFuncSetAttribute(kernel_of(t, t->f8 && form == 0), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
        if (e != cudaSuccess) return fail("cudaFuncSetAttribute", e);
    }
    return R3_OK;
}

bool tc_accept(const r3_fit_state& st, const float* sf2, const unsigned* wmax, unsigned xamax)
{
    auto value = [](unsigned bits) {
        float v;
        memcpy(&v, &bits, sizeof(v));
        return v;
    };
    if (!(value(xamax) <= kMaxScaled)) return false;   // scaled coordinates beyond the FP16 planes
    for (int g = 0; g < st.batch; ++g) {
        int sw, sk;
        operand_scales(value(wmax[g]), sf2[g], ops_of(&st)->f8, sw, sk);
        if (!(value(wmax[g]) > 0.f) || sw < -60 || sw > 60 || sk < -60 || sk > 60) return false;   // degenerate scales
    }
    return true;
}

void tc_info(const r3_gp* gp, int* info)
{
    const TensorOperands* t = ops_of(gp);
    for (int i = 0; i < 8; ++i) info[i] = 0;
    if (!t) return;
    info[0] = 256; info[1] = t->P; info[2] = t->DP; info[3] = t->NP;
    info[4] = t->G; info[5] = t->ws; info[6] = t->pair ? 0 : 1; info[7] = t->f8 ? 1 : 0;
}

// How many units a tile's pairs of strips are shared out to.  A pool of few tiles leaves SMs idle, and one of a few waves its
// last wave: the parts of a tile are scored by different CTAs and the last of them adds the sums up.  The choice minimises
// waves x the longest part, a pair of strips counted as its chunks of k* and a unit as kUnitChunks more (prologue, drain of the
// pipeline, epilogue).  It depends on the whole pool, not on the piece a launch covers, so that a pool scored in pieces gets the
// sums of one scored at once.
constexpr int kUnitChunks = 8;
static int plan_splits(const TensorOperands* t, long long tiles, int sms, unsigned char* cut)
{
    const int nc = t->NP / KC;
    auto chunks = [&](int p) { return std::min(8 * (p + 1), nc); };
    cut[0] = 0;
    cut[1] = (unsigned char)t->P;
    long long all = 0;
    for (int p = 0; p < t->P; ++p) all += chunks(p);
    int best = 1;
    if (tiles >= 16ll * sms || t->pair) return best;
    long long best_cost = (tiles + sms - 1) / sms * (all + kUnitChunks);
    best_cost -= best_cost / 20;   // sharing out has to gain something
    for (int k = 2; k <= std::min(t->P, kMaxSplits); ++k) {
        unsigned char c[kMaxSplits + 2] = {0};
        long long longest = 0, done = 0;
        int p = 0;
        for (int i = 0; i < k; ++i) {   // pairs up to the next k-th of the chunks, at least one, one left for each part behind
            const long long from = done, goal = all * (i + 1) / k;
            do done += chunks(p++);
            while (p < t->P - (k - 1 - i) && done + chunks(p) / 2 <= goal);
            if (i == k - 1)
                for (; p < t->P; ++p) done += chunks(p);
            c[i + 1] = (unsigned char)p;
            longest = std::max(longest, done - from);
        }
        const long long cost = (tiles * k + sms - 1) / sms * (longest + kUnitChunks);
        if (cost < best_cost) {
            best_cost = cost;
            best = k;
            for (int i = 0; i <= k; ++i) cut[i] = c[i];
        }
    }
    return best;
}

static int device_sms(int device)
{
    int sms = 148;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    return sms;
}

// guard's workspace, then the tiles' largest EI (one of each 32 rows), the sums of split tiles and their counters
static size_t max_bytes(const r3_gp* gp, long long m) { return ((size_t)score_tc_tiles(gp, m) * sizeof(float4) + 511) & ~(size_t)255; }
// With FP8 cross terms, the tiles that are scored first and decide for the pool: what is left over when the pool is cut into
// whole waves, so that the rest is whole waves, but at least a quarter of one.  Their pairs of strips are shared out over all
// SMs.  (A whole wave of tiles: 0.8 ms of the 10.5 ms of a round at n = 4096 whose 512 tiles are then scored with FP16 cross
// terms, 0.36 ms now; 1,048,576 candidates that keep them 55 waves and a third instead of 56.)
static long long pilot_tiles(const r3_gp* gp, long long m, int sms)
{
    const long long tiles = score_tc_tiles(gp, m);
    return std::min(tiles, std::max<long long>(sms / 4, tiles % sms));
}
// tiles times parts whose sums a call has to hold
static size_t split_slots(const r3_gp* gp, long long m)
{
    unsigned char cut[kMaxSplits + 2];
    const TensorOperands* t = ops_of(gp);
    const int sms = device_sms(gp->device);
    const long long tiles = score_tc_tiles(gp, m), first = t->f8 ? pilot_tiles(gp, m, sms) : 0;
    const int splits = plan_splits(t, tiles, sms, cut), first_splits = t->f8 ? plan_splits(t, first, sms, cut) : 1;
    return std::max<size_t>(splits > 1 ? tiles * splits : 0, first_splits > 1 ? first * first_splits : 0);
}
static size_t split_bytes(const r3_gp* gp, long long m)
{
    const size_t slots = split_slots(gp, m);
    return slots ? slots * 4 * TILE_M * sizeof(double) + score_tc_tiles(gp, m) * sizeof(int4) + 256 : 0;
}
size_t score_tc_workspace_bytes(const r3_gp* gp, long long m) { return guard_workspace_bytes(gp, m) + max_bytes(gp, m) + split_bytes(gp, m); }

static float* tile_max_of(const r3_gp* gp, long long m, void* ws)   // nullptr: the paired kernel leaves none
{
    if (ops_of(gp)->pair) return nullptr;
    return reinterpret_cast<float*>(((uintptr_t)ws + guard_workspace_bytes(gp, m) + 255) & ~(uintptr_t)255);
}

r3_status_t score_tc(r3_gp* gp, const float* Xcand, long long m, float* mu, float* sigma, float* ei, void* ws,
                     size_t ws_bytes, cudaStream_t stream)
{
    return score_tc_part(gp, Xcand, m, mu, sigma, ei, ws, ws_bytes, 0, -1, true, stream);
}

long long score_tc_tiles(const r3_gp* gp, long long m) { return (m + TILE_M - 1) / TILE_M * gp->batch; }

long long score_tc_first_tiles(const r3_gp* gp, long long m) { return ops_of(gp)->f8 ? pilot_tiles(gp, m, device_sms(gp->device)) : 0; }

bool score_tc_can_split(const r3_gp* gp) { return ops_of(gp) != nullptr && !ops_of(gp)->pair; }

r3_status_t score_tc_guard(r3_gp* gp, const float* Xcand, long long m, float* mu, float* sigma, float* ei, void* ws,
                           cudaStream_t stream)
{
    return guard_and_rescue(gp, Xcand, m, guard_carve(gp, m, ws), mu, sigma, ei, tile_max_of(gp, m, ws), (m + TILE_M - 1) / TILE_M, false, stream);
}

r3_status_t score_tc_part(r3_gp* gp, const float* Xcand, long long m, float* mu, float* sigma, float* ei, void* ws,
                          size_t ws_bytes, long long tile_begin, long long tile_end, bool guard, cudaStream_t stream)
{
    TensorOperands* t = ops_of(gp);
    if (!t) {
        set_error("the tensor-core engine does not serve this handle");
        return R3_ERR_UNSUPPORTED;
    }
    if (ws_bytes < score_tc_workspace_bytes(gp, m)) {
        set_error("internal: tensor workspace too small");
        return R3_ERR_INVALID_ARG;
    }
    const GuardBuffers gb = guard_carve(gp, m, ws);
    TcParams prm;
    prm.xcand = Xcand;
    prm.m = m;
    prm.batch = gp->batch;
    prm.d = gp->d;
    prm.mu = mu;
    prm.sigma = sigma;
    prm.ei = ei;
    prm.err_mu = gb.err_mu;
    prm.err_q = gb.err_q;
    prm.centre = t->centre;
    prm.scale = t->scale;
    prm.xt = t->xt;
    prm.xs32 = t->xs32;
    prm.xnorm = t->xnorm;
    prm.xnmax = t->xnmax;
    prm.alpha = t->alpha;
    prm.wt = t->wt;
    prm.kscale = t->kscale;
    prm.vinv2 = t->vinv2;
    prm.wt_gp_stride = t->wt_gp_stride;
    prm.sf2 = gp->sf2_d;
    prm.best = gp->best_d;
    prm.wnorm = gp->wnorm_d;
    prm.DP = t->DP;
    prm.NP = t->NP;
    prm.P = t->P;
    prm.ws = t->ws;
    prm.parts = t->parts;
    prm.S = t->S;
    prm.nc = t->NP / KC;
    prm.zb = t->zb;
    prm.xs = t->xs;
    prm.rsqrt_dp = 1.0 / sqrt((double)round_up(gp->d, 16));
    prm.status = gp->status_d;
    prm.tiles_per_gp = (m + TILE_M - 1) / TILE_M;
    prm.total_tiles = prm.tiles_per_gp * gp->batch;
    prm.tile_begin = 0;
    prm.wait_limit = gp->wait_limit_cycles;
    prm.withhold_w = gp->withhold_w;
    gp->withhold_w = -1;   // one call only
    if (tile_end >= 0) {   // a range of the pool's tiles (the caller runs the guard once, after the last range)
        prm.tile_begin = tile_begin;
        prm.total_tiles = tile_end < prm.total_tiles ? tile_end : prm.total_tiles;
    }
    const long long launch_tiles = prm.total_tiles - prm.tile_begin;
    if (launch_tiles <= 0) return R3_OK;
    prm.zero = gb.count;
    prm.zero_ints = guard_zero_ints(gp);
    prm.mode = nullptr;
    prm.want_mode = 0;
    const int sms = device_sms(gp->device);
    prm.splits = plan_splits(t, prm.tiles_per_gp * gp->batch, sms, prm.cut);
    prm.tile_max = tile_max_of(gp, m, ws);
    prm.partial = nullptr;
    prm.arrived = nullptr;
    if (const size_t slots = t->pair ? 0 : split_slots(gp, m)) {
        uintptr_t at = (uintptr_t)ws + guard_workspace_bytes(gp, m) + max_bytes(gp, m);
        at = (at + 255) & ~(uintptr_t)255;
        prm.partial = reinterpret_cast<double*>(at);
        prm.arrived = reinterpret_cast<int*>(prm.partial + slots * 4 * TILE_M);
    }
    prof_begin(gp, stream);
    if (t->pair) {
        const r3_status_t st = launch_tc_pair(t, prm, sms, stream);
        if (st != R3_OK) return st;
    } else {
        // planned: the tiles that the split is planned for, where it is not the whole pool; 0: no split
        auto launch = [&](bool f8, long long begin, long long end, int want_mode, long long planned = -1) -> r3_status_t {
            TcParams q = prm;
            if (planned >= 0) q.splits = plan_splits(t, planned, sms, q.cut);
            q.tile_begin = begin;
            q.total_tiles = end;
            q.mode = want_mode < 0 ? nullptr : gb.mode;
            q.want_mode = want_mode;
            if (t->f8 && !f8) {
                q.wt = t->wt16;
                q.vinv2 = t->vinv2_16;
            }
            if (q.splits > 1) R3_CUDA_TRY(cudaMemsetAsync(q.arrived, 0, sizeof(int4) * (end - begin), stream));
            void (*kernel)(const TcParams) = kernel_of(t, f8);
            R3_LAUNCH(kernel, (unsigned)std::min<long long>((end - begin) * q.splits, sms), kThreads, t->smem_bytes, stream, q);
            return R3_OK;
        };
        const long long begin = prm.tile_begin, end = prm.total_tiles;
        r3_status_t st = R3_OK;
        if (!t->f8) {
            st = launch(false, begin, end, -1);
        } else {
            // The FP8 cross terms save a fifth of the time where the posterior is tame and send most of a pool to the FP64
            // pass where it is not (few features, long lengthscales): 65,536 candidates at n = 4096 with 41,604 recomputed
            // 41.6 ms, with FP16 cross terms and none recomputed 4.1 ms.  So the pool's first tiles, as they lie in
            // memory, are scored with them, a test of it (pilot_kernel) decides on the device for the whole pool, and of the two
            // launches for the rest (for all of it, in the FP16 form) one returns at once.  A first part costs no more alone
            // than as part of the whole (pilot_tiles).
            const long long first = pilot_tiles(gp, m, sms);   // of the whole pool, whatever this launch covers
            long long rest = begin;
            if (begin == 0) {
                rest = std::min(end, first);
                st = launch(true, 0, rest, -1, first);
                // candidates of the first `rest` tiles that lie together in memory: whole GPs and a part of the next
                const long long whole = rest / prm.tiles_per_gp, part = std::min(m, rest % prm.tiles_per_gp * TILE_M);
                if (st == R3_OK) st = guard_pilot(gp, m, whole * m + part, gb, mu, sigma, ei, stream);
            }
            // Where the first tiles leave whole waves, sharing out only costs (25,000 candidates at n = 2000: 412 us shared out,
            // 401 us not); otherwise the rest is shared out as the pool would be (19,000, less than a wave: 377 us not, 364 us so).
            const bool whole = (prm.tiles_per_gp * gp->batch - first) % sms == 0;
            if (st == R3_OK && rest < end) st = launch(true, rest, end, t->wt16 ? 0 : -1, whole ? 0 : -1);
            if (st == R3_OK && t->wt16) st = launch(false, begin, end, 1);
        }
        if (st != R3_OK) return st;
    }
    prof_end(gp, stream);
    if (!guard) return R3_OK;
    return guard_and_rescue(gp, Xcand, m, gb, mu, sigma, ei, prm.tile_max, prm.tiles_per_gp, false, stream);
}

}  // namespace r3
