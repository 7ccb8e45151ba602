// vc_adj.cuh -- product of one row of the adjoint's matrix P_pi^T (AdjRows), shared by the
// BiCGSTAB solve, the fixed-point sweep and the FP64 residual.
#pragma once

#include "vc_internal.cuh"

namespace vc {

// sum_j val_j x[col_j] of row y in order of source, fused multiply-adds; up to B entries'
// columns, values and gathers are in flight before the first of them is added (rows of up to
// 2C entries and more per host occur: with one at a time a sweep of a 1,000-slot model took
// 287 us, its residual 610).
template <int B, typename T>
__device__ __forceinline__ T adj_row_dot(const AdjRows& t, const T* val, int y, const T* x) {
    const int n = __ldg(t.cnt + y);
    const int64_t lo = __ldg(t.base + (y >> 5)) + (y & 31);
    const int32_t* cp = t.col + lo;
    const T* vp = val + lo;
    T acc = T(0);
    for (int j0 = 0; j0 < n; j0 += B, cp += 32 * B, vp += 32 * B) {
        T w[B], g[B];
#pragma unroll
        for (int u = 0; u < B; u++) {
            if (j0 + u < n) {
                w[u] = __ldg(vp + 32 * u);
                g[u] = x[__ldg(cp + 32 * u)];
            }
        }
#pragma unroll
        for (int u = 0; u < B; u++)
            if (j0 + u < n) acc = fma(w[u], g[u], acc);
    }
    return acc;
}

}  // namespace vc
