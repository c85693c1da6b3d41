// Column sums of a projection's partial results, shared by the kernels that finish it.  The columns (up to 296) are cut
// into kFinishSlices ranges summed side by side, then the ranges are added in ascending order: a single thread per entry
// would wait for L2 some seventy times in a row (34 us at m = 256 and n = 8, where this takes 4).  Whoever finishes an
// entry with these two functions gets the same bits.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <type_traits>

namespace core {

constexpr int kFinishSlices = 8;

// p[0] + p[stride] + ... of `count` numbers, in ascending order, FIRST and then AT (4, 8 or 16) loads in flight at a time, and the last ones, fewer
// than that, together too: a loop unrolled by the compiler may fetch those one after the other, each a round trip to L2 (us: a decentralised
// step of 16 machines, d = 20000, m = 64: 86.4 -> 84.0).
template <int AT, int FIRST = AT, typename T>
__device__ __forceinline__ T sum_strided(const T *p, int count, int64_t stride) {
    T s = 0;
    auto batch = [&](auto size) {
        constexpr int N = decltype(size)::value;
        T v[N];
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __ldcg(p + i * stride);
#pragma unroll
        for (int i = 0; i < N; ++i) s += v[i];
        count -= N;
        p += N * stride;
    };
    if constexpr (FIRST > AT) {
#pragma unroll 1
        while (count >= FIRST) batch(std::integral_constant<int, FIRST>{});
    }
    while (count >= AT) batch(std::integral_constant<int, AT>{});
    T a[8], b[4], c[2], d = 0;
    if (AT > 8 && count & 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = __ldcg(p + i * stride);
        p += 8 * stride;
    }
    if (AT > 4 && count & 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = __ldcg(p + i * stride);
        p += 4 * stride;
    }
    if (count & 2) {
        c[0] = __ldcg(p);
        c[1] = __ldcg(p + stride);
        p += 2 * stride;
    }
    if (count & 1) d = __ldcg(p);
    if (AT > 8 && count & 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) s += a[i];
    }
    if (AT > 4 && count & 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) s += b[i];
    }
    if (count & 2) {
        s += c[0];
        s += c[1];
    }
    return count & 1 ? s + d : s;
}

// (Fewer at a time in kernels that want their registers for something else: the gossip of 17 to 32 machines spilled with sixteen: 1.2 us
// a step.)
template <int AT = 16, int FIRST = AT>
__device__ __forceinline__ float finish_slice(const float *partial, int chunks, int64_t total, int64_t idx, int slice) {
    const int begin = chunks * slice / kFinishSlices, end = chunks * (slice + 1) / kFinishSlices;
    return sum_strided<AT, FIRST>(partial + (int64_t)begin * total + idx, end - begin, total);
}

// The slices of an entry, `stride` floats apart.
__device__ __forceinline__ float finish_join(const float *slices, int stride) {
    float s = slices[0];
#pragma unroll
    for (int r = 1; r < kFinishSlices; ++r) s += slices[r * stride];
    return s;
}

}  // namespace core
