// Small kernels of the optimiser variants built on the round: the step rule of Algorithm 3's Option I
// (chosen on the device from the size of the combined messages) and the gossip averaging of
// Algorithm 5 (decentralised CORE-GD).  Everything here works on n x m or m numbers: microseconds.
#include "core_internal.h"
#include "core_sync.cuh"

namespace core {

namespace {

constexpr int kVarThreads = 256;

// p = sqrt((1/m) sum_j pbar_j^2) and h = min{ m / (16 r1), c H^-1/2 p^-1/2 d^-3/4 m^3/4 }.
// One CTA; thread t sums entries t, t + 256, ... in ascending order, the 256 partial sums are added in
// ascending order by thread 0: a fixed order, in double (m numbers, nothing to save in fp32).
__global__ void option1_step_kernel(const float * pbar, int m, double d, double r1, double H, double c,
                                    float *p_out, float *h_out) {
    grid_trigger();
    grid_wait();
    __shared__ double part[kVarThreads];
    double s = 0.0;
    for (int j = threadIdx.x; j < m; j += kVarThreads) s += (double)pbar[j] * (double)pbar[j];
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double total = 0.0;
    for (int r = 0; r < kVarThreads; ++r) total += part[r];
    const double p = sqrt(total / (double)m);
    const double first = (double)m / (16.0 * r1);
    // p = 0 (no gradient at all) makes the second term infinite: the first one decides
    const double second = c * rsqrt(H) * rsqrt(p) * pow(d, -0.75) * pow((double)m, 0.75);
    *h_out = (float)(first < second ? first : second);
    if (p_out) *p_out = (float)p;
}

// One gossip round: out[i][j] = sum_l W[i][l] in[l][j], l ascending.
__global__ void gossip_round_kernel(const float * W, const float * in, int n, int m,
                                    float *out) {
    grid_trigger();
    grid_wait();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y;
    if (j >= m) return;
    float s = 0.f;
    for (int l = 0; l < n; ++l) s = fmaf(W[(int64_t)i * n + l], in[(int64_t)l * m + j], s);
    out[(int64_t)i * m + j] = s;
}

// All gossip rounds of a step in one launch: a column of the messages never meets another one, so a CTA takes
// kGossipCols columns of all machines through every round in shared memory, W beside them.  Same products in the same
// order as gossip_round_kernel, hence the same bits.  Bound by latency (n multiply-adds and a barrier per round): twenty
// rounds of 16 machines took 46 us of launches (2.3 us each), here 4 us.
constexpr int kGossipCols = 8;
constexpr int kGossipMaxMachines = 128;               // W in 64 KB of shared memory
__global__ void gossip_rounds_kernel(const float * W, const float * in, int n, int m, int rounds,
                                     float *out) {
    grid_trigger();
    grid_wait();
    extern __shared__ float gossip_smem[];
    const int ldw = n + 1;                            // rows of W that are read together fall into different banks
    float *const weights = gossip_smem, *cur = weights + n * ldw, *nxt = cur + n * kGossipCols;
    const int tid = threadIdx.x, threads = blockDim.x;
    const int col = tid % kGossipCols, j = blockIdx.x * kGossipCols + col;
    for (int e = tid; e < n * n; e += threads) weights[(e / n) * ldw + e % n] = W[e];
    for (int i = tid / kGossipCols; i < n; i += threads / kGossipCols)
        cur[i * kGossipCols + col] = j < m ? in[(int64_t)i * m + j] : 0.f;
    __syncthreads();
    for (int r = 0; r < rounds; ++r) {
        for (int i = tid / kGossipCols; i < n; i += threads / kGossipCols) {
            float s = 0.f;
#pragma unroll 8
            for (int l = 0; l < n; ++l) s = fmaf(weights[i * ldw + l], cur[l * kGossipCols + col], s);
            nxt[i * kGossipCols + col] = s;
        }
        __syncthreads();
        float *const swap = cur;
        cur = nxt;
        nxt = swap;
    }
    if (j < m)
        for (int i = tid / kGossipCols; i < n; i += threads / kGossipCols) out[(int64_t)i * m + j] = cur[i * kGossipCols + col];
}

// spread[0] = max over machines i and vectors j of |P[i][j] - P[reader][j]| (a maximum: order-free).
__global__ void consensus_spread_kernel(const float * P, int n, int m, int reader, float *spread) {
    grid_trigger();
    grid_wait();
    __shared__ float part[kVarThreads];
    float worst = 0.f;
    for (int64_t e = threadIdx.x; e < (int64_t)n * m; e += kVarThreads)
        worst = fmaxf(worst, fabsf(P[e] - P[(int64_t)reader * m + e % m]));
    part[threadIdx.x] = worst;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int r = 1; r < kVarThreads; ++r) worst = fmaxf(worst, part[r]);
    *spread = worst;
}

}  // namespace

cudaError_t launch_option1_step(const float *pbar, int32_t m, int64_t d, double r1, double H, double c, float *p_out,
                                float *h_out, cudaStream_t stream) {
    return launch_chained(true, option1_step_kernel, dim3(1), dim3(kVarThreads), 0, stream, pbar, m, (double)d, r1, H, c, p_out, h_out);
}

cudaError_t launch_gossip_round(const float *W, const float *in, int32_t n, int32_t m, float *out, cudaStream_t stream) {
    dim3 grid((unsigned)((m + 127) / 128), (unsigned)n);
    return launch_chained(true, gossip_round_kernel, grid, dim3(128), 0, stream, W, in, n, m, out);
}

cudaError_t launch_gossip_rounds(const float *W, float *P, int32_t n, int32_t m, int32_t rounds, float *scratch, float **result,
                                 cudaStream_t stream) {
    *result = P;
    if (rounds <= 0) return cudaSuccess;
    if (n <= kGossipMaxMachines) {
        const size_t smem = ((size_t)n * (n + 1) + 2 * (size_t)n * kGossipCols) * sizeof(float);
        const int rows = n < 64 ? n : 64;
        *result = scratch;
        return launch_chained(true, gossip_rounds_kernel, dim3((m + kGossipCols - 1) / kGossipCols), dim3(kGossipCols * rows), smem, stream, W,
                              P, n, m, rounds, scratch);
    }
    for (int32_t r = 0; r < rounds; ++r) {
        cudaError_t e = launch_gossip_round(W, P, n, m, scratch, stream);
        if (e != cudaSuccess) return e;
        float *const swap = P;
        P = scratch;
        scratch = swap;
    }
    *result = P;
    return cudaSuccess;
}

cudaError_t launch_consensus_spread(const float *P, int32_t n, int32_t m, int32_t reader, float *spread,
                                    cudaStream_t stream) {
    return launch_chained(true, consensus_spread_kernel, dim3(1), dim3(kVarThreads), 0, stream, P, n, m, reader, spread);
}

}  // namespace core
