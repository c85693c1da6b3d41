// Column sums of a projection's partial results, shared by the kernels that finish it.  The columns (up to 296) are cut
// into kFinishSlices ranges summed side by side, then the ranges are added in ascending order: a single thread per entry
// would wait for L2 some seventy times in a row (34 us at m = 256 and n = 8, where this takes 4).  Whoever finishes an
// entry with these two functions gets the same bits.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace core {

constexpr int kFinishSlices = 8;

// p[0] + p[stride] + ... of `count` numbers, in ascending order, eight loads in flight at a time also where fewer are left: a loop
// unrolled by the compiler fetches its last up to seven one after the other, each a round trip to L2 (us: a round of
// four machines, d = 4096, m = 16: 8.2 -> 7.1; a decentralised step of 16 machines, d = 20000, m = 64: 86.4 -> 84.0).
template <typename T>
__device__ __forceinline__ T sum_strided(const T *p, int count, int64_t stride) {
    T s = 0;
    for (int c = 0; c < count; c += 8, p += 8 * stride) {
        T v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = c + i < count ? __ldcg(p + i * stride) : (T)0;
#pragma unroll
        for (int i = 0; i < 8; ++i) s += v[i];
    }
    return s;
}

__device__ __forceinline__ float finish_slice(const float *partial, int chunks, int64_t total, int64_t idx, int slice) {
    const int begin = chunks * slice / kFinishSlices, end = chunks * (slice + 1) / kFinishSlices;
    return sum_strided(partial + (int64_t)begin * total + idx, end - begin, total);
}

// The slices of an entry, `stride` floats apart.
__device__ __forceinline__ float finish_join(const float *slices, int stride) {
    float s = slices[0];
#pragma unroll
    for (int r = 1; r < kFinishSlices; ++r) s += slices[r * stride];
    return s;
}

}  // namespace core
