// vc_grid.cuh -- grid barrier of the resident kernels, their launch and the stopping test of
// the value-iteration loops among them.
//
// The kernels are cooperative launches of at most the resident grid, so every block of a
// barrier runs; each wait still has an iteration limit, after which the block gives up, the
// kernel flags a timeout and returns.
#pragma once

#include <math.h>

#include "vc_internal.cuh"

namespace vc {

constexpr unsigned int kBarrierPolls = 1u << 22;  // a few seconds

// Poll limit of a launch's barrier waits from a control block's spin_limit (the handle's cap + 1,
// 0 without one).
__host__ __device__ inline unsigned int barrier_polls(long long spin_limit) {
    return spin_limit > 0 && spin_limit - 1 < (long long)kBarrierPolls ? (unsigned int)(spin_limit - 1) : kBarrierPolls;
}

// A counter that only grows during a launch (the host clears it before): barrier n is complete
// once it reaches n x blocks.  Memory written before the barrier by any thread of the
// grid is visible after it to every thread (thread 0's fences, ordered by the block's own
// barriers; the acquire also drops stale L1 lines, so plain loads follow).
struct GridBarrier {
    unsigned int* count;
    unsigned int blocks, target;
    int* fail;           // shared: set once a wait gave up
    unsigned int limit;  // polls of a wait (barrier_polls)

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
            } while (v < target && ++polls < limit);
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

// A resident launch holds every SM, so kernels of other streams wait for its end: it ends itself
// after about 4 ms (8 M cycles at 2 GHz; the host reads the control block and goes on with another
// launch, some 30 us: under 1 %), at a sweep that all CTAs take from one word.  CTA 0 writes it two
// sweeps ahead: whoever still reads for the sweep before finds a number that it has not
// reached, and everyone has it after the next barrier.  Whole solves on one launch held the
// device for up to 0.25 s.
constexpr long long kLaunchCycles = 8'000'000;
constexpr long long kLaunchSweeps = 1 << 20;

struct LaunchEnd {
    long long* end;    // the control block's word
    long long* start;  // shared: clock64() at the launch (a register pair in every thread cost the
                       // stored-matrix loop 2 %)
    // Thread 0 of CTA 0, before its first barrier.
    __device__ __forceinline__ void open(long long k) {
        *start = clock64();
        *((volatile long long*)end) = k + kLaunchSweeps;
    }
    // The same thread at the start of sweep k (0-based).
    __device__ __forceinline__ void check(long long k) {
        if (clock64() - *start > kLaunchCycles && *((volatile long long*)end) > k + 2)
            *((volatile long long*)end) = k + 2;
    }
    __device__ __forceinline__ long long read() const { return *((volatile long long*)end); }
};

// Step 3's test on every thread of a CTA from the sweep's residual r and max|V'| vm:
// finish_block's decision, in the same order.  4 ulp(vm) is a power of two, so for vm
// above 2^-100 both sides of r < max(tol, 4 ulp) are compared in FP32 exactly (tol rounded
// up to FP32: r < tol iff r < that).
struct LoopVerdict {
    double tol;
    float tol32, best;
    int since;
    long long max_sweeps;
    __device__ int operator()(float r, float vm, long long k) {
        bool below;
        if (vm >= 0x1p-100f) {
            const float ulp4 = __uint_as_float((fbits(vm) & 0x7f800000u) - (21u << 23));
            below = r < tol32 || r < ulp4;
        } else {
            int e = 0;
            frexpf(vm, &e);
            const double ulp = vm > 0.0f ? ldexp(1.0, e - 24) : 0.0;
            below = (double)r < fmax(tol, 4.0 * ulp);
        }
        int done = 0;
        if (below) {
            done = 1;
        } else if (r < best) {
            best = r;
            since = 0;
        } else if (++since >= kStallSweeps) {
            done = 3;
        }
        if (!done && k >= max_sweeps) done = 2;
        return done;
    }
};

// Cooperative launch; *launched = false (and nothing enqueued) when the grid cannot be
// resident at once on this device.  The caller keeps `turn` until it has read the result.
template <typename... Args>
int launch_resident(const void* kern, int grid, int threads, size_t smem, cudaStream_t st, ResidentTurn& turn,
                    int num_sms, bool* launched, Args... args) {
    void* ptrs[] = {(void*)&args...};
    turn.take(grid, num_sms);
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
