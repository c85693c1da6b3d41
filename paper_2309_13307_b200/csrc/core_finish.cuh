// Column sums of a projection's partial results, shared by the kernels that finish it.  The columns (up to 296) are cut
// into kFinishSlices ranges summed side by side, then the ranges are added in ascending order: a single thread per entry
// would wait for L2 some seventy times in a row (34 us at m = 256 and n = 8, where this takes 4).  Whoever finishes an
// entry with these two functions gets the same bits.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace core {

constexpr int kFinishSlices = 8;

__device__ __forceinline__ float finish_slice(const float *partial, int chunks, int64_t total, int64_t idx, int slice) {
    const int begin = chunks * slice / kFinishSlices, end = chunks * (slice + 1) / kFinishSlices;
    float s = 0.f;
#pragma unroll 8
    for (int c = begin; c < end; ++c) s += __ldcg(partial + (int64_t)c * total + idx);
    return s;
}

// The slices of an entry, `stride` floats apart.
__device__ __forceinline__ float finish_join(const float *slices, int stride) {
    float s = slices[0];
#pragma unroll
    for (int r = 1; r < kFinishSlices; ++r) s += slices[r * stride];
    return s;
}

}  // namespace core
