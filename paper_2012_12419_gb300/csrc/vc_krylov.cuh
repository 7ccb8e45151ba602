// vc_krylov.cuh -- BiCGSTAB correction solve of the refinement: scalars, stages and entry.
//
// The mixed-precision refinement solves, for a fixed policy pi, the correction equation
// (I - gamma P_pi) e = r, where r = T_pi V64 - V64 is the FP64 policy residual stored in
// FP32.  Plain fixed-point sweeps e <- r + gamma P_pi e converge at rate gamma per sweep;
// BiCGSTAB (H. A. van der Vorst, SIAM J. Sci. Stat. Comput. 13(2), 1992), unpreconditioned,
// in FP32, reaches the same stopping test (max |r - (I - gamma P_pi) e| below the target)
// with fewer products by the matrix on these uniformised chains.
//
// One iteration: p update, v = A p (with <b, v>), s = r - alpha v, t = A s (with <t, s>,
// <t, t>), and the x / r update (with <b, r> and max |r|).  The reductions run in a fixed
// order, so a solve is deterministic.
#pragma once

#include "vc_internal.cuh"

namespace vc {

struct KrylovCtl {
    double rho;       // <b, r> of the current residual (b is the shadow residual)
    double alpha, omega, beta;
    double target;    // stop once max |r| < target (raised to 2^-18 max |b| by the first stage)
    float rmax;       // max |r| after the last iteration
    int done;         // 0 running, 1 converged, 2 iteration cap, 5 breakdown
    int iter, max_iter;
    unsigned int arrivals;  // grid barrier of the resident kernel: arrivals since the launch
    int fault;              // set by a block whose barrier wait gave up
    long long spin_limit;   // polls + 1 of a barrier wait (0: the default)
    long long launch_end;   // iterations at which the launch ends (LaunchEnd)
};

enum KrylovStage : int { kKrInit = 0, kKrV = 1, kKrT = 2, kKrX = 3 };

// Partial sums of the resident kernel: a stage stores a CTA's (two sums and a maximum), passes
// one grid barrier, and every CTA reads all of them.  A late CTA may still read stage T's
// while an early one stores stage X's, as no barrier lies between the two (the x / r update
// touches only a CTA's own states), so these two use different sets.  Before every other
// stage the product's first barrier separates the last readers from the next writers.
constexpr int kKrPartSets = 2;
constexpr int kKrPartValues = 3;  // per CTA and set
__host__ __device__ constexpr int kr_part_set(int stage) { return stage % kKrPartSets; }
static_assert(kr_part_set(kKrT) != kr_part_set(kKrX), "no barrier between the readers of T and the writers of X");

// Block-wide sum over NT threads in a fixed order; result valid in thread 0.
template <int NT>
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double part[NT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) part[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = (l < NT / 32) ? part[l] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    }
    __syncthreads();
    return r;
}

// Entries of one BiCGSTAB vector in the handle's work space: vectors start on 256 bytes.
inline size_t krylov_stride(int64_t n) { return ((size_t)n + 63) & ~(size_t)63; }

// BiCGSTAB solve of (I - gamma P_pi) x = b from x = 0 until max |b - (I - gamma P_pi) x|
// (the recurrence residual) is below target or max_iter iterations; *products counts the
// products by the matrix, *converged reports whether the target was met (a breakdown or
// the iteration cap leave it false; the caller then falls back to fixed-point sweeps).
int krylov_correct(Mdp* m, const int32_t* pi, const float* b, float* x, double target, long long max_iter,
                   cudaStream_t st, long long* products, bool* converged);

}  // namespace vc
