// FP64 building blocks shared by the kernels that work in double precision: the tensor path's 8x8x4 product,
// asynchronous copies into shared memory, and the barrier of a cooperatively launched grid.
//
// Measured on B200: FP64 fused multiply-adds and mma.m8n8k4.f64 share one peak (36-37 TFLOP/s), but the matrix
// instruction reads its operands from shared memory a quarter as often, and a plain C = A B^T of 4096^3 with
// 64x64 tiles, 16-deep stages and three of them in flight runs at 33 TFLOP/s where the 4x4 register tiling of
// scalar multiply-adds stays at 14.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "r3_internal.cuh"

namespace r3 {

// c (8x8: lane l holds row l / 4, columns 2 (l % 4) + {0, 1}) += a (row l / 4, k = l % 4) * b (k = l % 4, column l / 4)
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                 : "+d"(c[0]), "+d"(c[1])
                 : "d"(a), "d"(b));
}

// 16 bytes from global to shared memory, asynchronously; zeros when !valid (nothing is read then)
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid = true)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Leading dimension (doubles) of a 16-deep operand stage: 20 = 4 mod 16 keeps the fragment reads of mma.m8n8k4
// (four consecutive k of eight rows per warp, half a warp at a time) on sixteen different 8-byte banks.
constexpr int kStageLd = 20;

__device__ __forceinline__ unsigned load_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Barrier over `blocks` blocks (grid_barrier: all) of a cooperatively launched grid.  `counter` starts at zero and only grows;
// `target` is the caller's running count.  Bounded like every device-side wait: when it runs out the status word gets
// DEV_TIMEOUT and false is returned, on which the block leaves the kernel.
__device__ __forceinline__ bool team_barrier(unsigned* counter, unsigned& target, unsigned blocks, int* status,
                                             const WaitRule& rule)
{
    bool ok = true;
    __syncthreads();
    target += blocks;
    if (threadIdx.x == 0) {
        __threadfence();
        if (!(rule.withhold && blockIdx.x == 0)) atomicAdd(counter, 1u);
        if (load_acquire(counter) < target) {
            const long long t0 = clock64();
            while (load_acquire(counter) < target) {
                if (clock64() - t0 > rule.cycles) {
                    atomicOr(status, DEV_TIMEOUT);
                    ok = false;
                    break;
                }
            }
        }
    }
    return __syncthreads_and(ok);
}
__device__ __forceinline__ bool grid_barrier(unsigned* counter, unsigned& target, int* status, const WaitRule& rule)
{
    return team_barrier(counter, target, gridDim.x, status, rule);
}

}  // namespace r3
