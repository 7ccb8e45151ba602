// vc_sell.cuh -- layout of a slice record of the sliced copy (vc_sell.cu).
#pragma once

#include "vc_internal.cuh"

namespace vc {

constexpr int kSellC = 32;  // states of a slice

__host__ __device__ inline long long round128(long long x) { return (x + 127) & ~127LL; }

// Byte offsets inside a slice record with `rows` rows of 32 entries.
struct RecLayout {
    int R, scale, col;
    long long val, bytes;
};

__host__ __device__ inline RecLayout rec_layout(int A, long long rows, int vt, bool has_scale) {
    RecLayout L;
    L.R = 256;
    L.scale = L.R + 128 * A;
    L.col = L.scale + (has_scale ? 128 * A : 0);
    L.val = L.col + 128LL * rows;
    L.bytes = L.val + round128(32LL * vt * rows);
    return L;
}

// The same from a stored record's header, in offsets of type I: int for a record in the shared-
// memory ring (a BF16 ring sweep of 12.5 M states takes 1,171 us with these, 1,337 with the
// 64-bit layout above formed for each action), long long for one in global memory, where a
// single long row makes a record of any size (its columns reach 2^31 bytes at 16.8 M rows).
template <typename I>
struct RecAt {
    int rows;
    I scale, col, val;
};

template <typename I>
__host__ __device__ __forceinline__ RecAt<I> rec_at(const unsigned char* rec, int A, bool has_scale) {
    RecAt<I> p;
    p.rows = reinterpret_cast<const int32_t*>(rec)[A];
    p.scale = 256 + 128 * A;
    p.col = p.scale + (has_scale ? 128 * A : 0);
    p.val = p.col + (I)128 * p.rows;
    return p;
}

}  // namespace vc
