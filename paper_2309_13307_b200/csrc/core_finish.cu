// Finishing a projection: the column sums of its partial results, and the mean message over the machines.
// In a unit of its own: the driver loads a unit's code as one when its first kernel is launched, and every projection kernel
// is finished by these.  Beside the scalar projection (2.8 MB of instances) they made a process's first round load that too:
// first core_project of one machine 2.9 ms -> 1.6, first core_round of eight at d = 4e6 4.3 ms -> 2.3.
#include "core_finish.cuh"
#include "core_internal.h"
#include "core_sync.cuh"

namespace core {

namespace {

// Few columns: one per slice, without the loops (us, 30 machines, d = 2000, m = 2500, eight columns: projection
// 19.8 -> 19.3, round 36.6 -> 35.9).
template <int AT>
__device__ __forceinline__ float any_slice(const float *partial, int chunks, int64_t total, int64_t idx, int slice) {
    if (chunks > kFinishSlices) return finish_slice<AT>(partial, chunks, total, idx, slice);
    const int begin = chunks * slice / kFinishSlices, end = chunks * (slice + 1) / kFinishSlices;
    return begin < end ? 0.f + __ldcg(partial + (int64_t)begin * total + idx) : 0.f;
}

__global__ void finish_project_kernel(const float *__restrict__ partial, int chunks, int n, int m,
                                      float *__restrict__ P, int accumulate) {
    grid_trigger();
    grid_wait();
    __shared__ float slices[kFinishSlices][32];
    const int64_t idx = (int64_t)blockIdx.x * 32 + threadIdx.x;
    const int64_t total = (int64_t)n * m;
    slices[threadIdx.y][threadIdx.x] = idx < total ? any_slice<16>(partial, chunks, total, idx, threadIdx.y) : 0.f;
    __syncthreads();
    if (threadIdx.y != 0 || idx >= total) return;
    const float s = finish_join(&slices[0][threadIdx.x], 32);
    P[idx] = accumulate ? P[idx] + s : s;
}

__global__ void aggregate_kernel(const float *__restrict__ P, int n, int m, float *__restrict__ pbar) {
    grid_trigger();
    grid_wait();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    pbar[j] = sum_strided<16>(P + j, n, m) / (float)n;
}

// Both of the above in one launch for a single group of machines whose messages nobody asks for:
// the same sums in the same order, so pbar is bitwise what the two kernels give.
// A CTA takes eight vectors, so that sixteen machines' slices are in flight together (32 vectors and four machines: 9.3 us
// for 22 machines, 232 vectors).  Eight loads at a time, for two CTAs per SM: with sixteen (40 registers) there is room for one, and 16 machines,
// d = 3368, m = 2210 took two waves (the round 38.9 -> 41.0 us).
constexpr int kFinishMachines = 16;
constexpr int kFinishVectors = 8;
__global__ void __launch_bounds__(kFinishMachines * kFinishSlices * kFinishVectors, 2)
finish_aggregate_kernel(const float *__restrict__ partial, int chunks, int n, int m, float *__restrict__ pbar) {
    grid_trigger();
    grid_wait();
    __shared__ float slices[kFinishMachines][kFinishSlices][kFinishVectors];
    const int lane = threadIdx.x, slice = threadIdx.y, row = threadIdx.z;
    const int j = blockIdx.x * kFinishVectors + lane;
    const int64_t total = (int64_t)n * m;
    float sum = 0.f;                    // kept by the first kFinishVectors threads
    for (int i0 = 0; i0 < n; i0 += kFinishMachines) {
        const int i = i0 + row;
        slices[row][slice][lane] = i < n && j < m ? any_slice<8>(partial, chunks, total, (int64_t)i * m + j, slice) : 0.f;
        __syncthreads();
        if (slice == 0 && row == 0)
            for (int r = 0; r < kFinishMachines && i0 + r < n; ++r) sum += finish_join(&slices[r][0][lane], kFinishVectors);
        __syncthreads();
    }
    if (slice == 0 && row == 0 && j < m) pbar[j] = sum / (float)n;
}

}  // namespace

cudaError_t launch_finish_project(const float *partial, int chunks, int32_t n, int32_t m, float *P,
                                  bool accumulate, cudaStream_t stream) {
    const int64_t total = (int64_t)n * m;
    return launch_chained(true, finish_project_kernel, dim3((unsigned)((total + 31) / 32)), dim3(32, kFinishSlices), 0, stream, partial,
                          chunks, n, m, P, accumulate ? 1 : 0);
}

cudaError_t launch_finish_aggregate(const float *partial, int chunks, int32_t n, int32_t m, float *pbar,
                                    cudaStream_t stream) {
    const int rows = n < kFinishMachines ? n : kFinishMachines;
    return launch_chained(true, finish_aggregate_kernel, dim3((m + kFinishVectors - 1) / kFinishVectors),
                          dim3(kFinishVectors, kFinishSlices, rows), 0, stream, partial, chunks, n, m, pbar);
}

cudaError_t launch_aggregate(const float *P, int32_t n, int32_t m, float *pbar, cudaStream_t stream) {
    const int threads = 128;
    return launch_chained(true, aggregate_kernel, dim3((m + threads - 1) / threads), dim3(threads), 0, stream, P, n, m, pbar);
}

}  // namespace core
