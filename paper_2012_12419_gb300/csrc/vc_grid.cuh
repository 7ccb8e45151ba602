// vc_grid.cuh -- grid barrier of the resident kernels and their launch.
//
// The kernels are cooperative launches of at most the resident grid, so every block of a
// barrier runs; each wait still has an iteration limit, after which the block gives up, the
// kernel flags a timeout and returns.
#pragma once

#include "vc_internal.cuh"

namespace vc {

constexpr unsigned int kBarrierPolls = 1u << 22;  // a few seconds

// A counter that only grows during a launch (the host clears it before): barrier n is complete
// once it reaches n x blocks.  Memory written before the barrier by any thread of the
// grid is visible after it to every thread (thread 0's fences, ordered by the block's own
// barriers; the acquire also drops stale L1 lines, so plain loads follow).
struct GridBarrier {
    unsigned int* count;
    unsigned int blocks, target;
    int* fail;  // shared: set once a wait gave up

    // Call after a __syncthreads that covers the block's writes; thread 0 holds the result
    // until the caller's next __syncthreads.
    __device__ __forceinline__ bool arrive_and_wait() {
        target += blocks;
        if (threadIdx.x == 0 && blocks > 1) {
            unsigned int v;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
            unsigned int polls = 0;
            do {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
            } while (v < target && ++polls < kBarrierPolls);
            if (v < target) *fail = 1;
        }
        __syncthreads();
        return *fail == 0;
    }
    __device__ __forceinline__ bool sync() {
        __syncthreads();
        return arrive_and_wait();
    }
};

// Cooperative launch; *launched = false (and nothing enqueued) when the grid cannot be
// resident at once on this device.
template <typename... Args>
int launch_resident(const void* kern, int grid, int threads, size_t smem, cudaStream_t st, bool* launched,
                    Args... args) {
    void* ptrs[] = {(void*)&args...};
    const cudaError_t e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)grid), dim3((unsigned)threads), ptrs, smem, st);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        *launched = false;
        return VC_OK;
    }
    if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchCooperativeKernel");
    count_launches(1);
    *launched = true;
    return VC_OK;
}

}  // namespace vc
