// Small kernels of the optimiser variants built on the round: the step rule of Algorithm 3's Option I
// (chosen on the device from the size of the combined messages) and the gossip averaging of
// Algorithm 5 (decentralised CORE-GD).  Everything here works on n x m or m numbers: microseconds.
#include "core_finish.cuh"
#include "core_internal.h"
#include "core_sync.cuh"

namespace core {

namespace {

constexpr int kVarThreads = 256;
constexpr int kSpreadThreads = 1024;

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

// Everything between the projection and the reconstruction of a decentralised step in one launch, for up to 64 machines: the
// messages from the projection's partial sums (the order of finish_project_kernel), all gossip rounds, the distance from
// consensus.  A column of the messages never meets another one, so a CTA takes kGossipCols columns of all machines through
// every round in shared memory; a thread holds one entry and its row of W in registers.  Same products in the same order
// as gossip_round_kernel (zero weights on zero rows at the end change nothing), hence the same bits.  Bound by latency: the
// loads of the partial sums (all threads, a slice of a message each), then NR multiply-adds in a row and a barrier per round.
// us of a step, 16 machines, d = 20000, m = 64, 20 rounds: finish, rounds with W in shared memory and distance as three
// launches 96.8, this one 91.5; 5 machines, d = 3000, m = 300, 30 rounds: 41.5 -> 34.4; 64 machines, d = 4096, m = 256, 20 rounds:
// 82.2 -> 63.1 (messages finished by a launch of their own).
constexpr int kGossipCols = 8;
constexpr int gossip_threads(int nr) { return nr <= 32 ? 1024 : 512; }      // that finish the messages: a row of W has to fit
template <int NR>
__global__ void __launch_bounds__(gossip_threads(NR))
gossip_step_kernel(const float *W, const float *partial, int chunks, const float *in, int n, int m, int rounds, float *out,
                   int reader, int *spread) {
    grid_trigger();
    constexpr int kLd = NR + 4;                       // an odd multiple of 16 bytes: columns fall into different banks
    __shared__ __align__(16) float buffers[2][kGossipCols][kLd];
    __shared__ float slices[NR * kGossipCols * kFinishSlices];
    __shared__ int worst;
    const int tid = threadIdx.x, col = tid % kGossipCols, i = tid / kGossipCols, j0 = blockIdx.x * kGossipCols, j = j0 + col;
    const int active = (n + 3) / 4 * 4 * kGossipCols; // threads with an entry, whole warps
    for (int e = tid; e < 2 * kGossipCols * kLd; e += blockDim.x) (&buffers[0][0][0])[e] = 0.f;
    if (tid == 0) worst = 0;
    grid_wait();
    float w[NR];
    if (tid < active) {
#pragma unroll
        for (int l = 0; l < NR; ++l) w[l] = i < n && l < n ? __ldcg(W + i * n + l) : 0.f;
    }
    if (partial) {
        const int entries = n * kGossipCols;
        for (int e = tid; e < entries * kFinishSlices; e += blockDim.x) {
            const int entry = e % entries, slice = e / entries, jj = j0 + entry % kGossipCols;
            slices[e] = jj < m ? finish_slice<NR >= 32 ? 4 : 8>(partial, chunks, (int64_t)n * m, (int64_t)(entry / kGossipCols) * m + jj, slice) : 0.f;
        }
        __syncthreads();
        if (tid < entries) buffers[0][col][i] = finish_join(slices + tid, entries);
    } else {
        __syncthreads();                              // the buffers are zero
        if (i < n && j < m) buffers[0][col][i] = __ldcg(in + (int64_t)i * m + j);
    }
    __syncthreads();
    if (tid >= active) return;
    int cur = 0;
    for (int r = 0; r < rounds; ++r, cur ^= 1) {
        const float4 *const column = reinterpret_cast<const float4 *>(buffers[cur][col]);
        float s = 0.f;
#pragma unroll
        for (int l = 0; l < NR / 4; ++l) {
            const float4 p = column[l];
            s = fmaf(w[4 * l], p.x, s);
            s = fmaf(w[4 * l + 1], p.y, s);
            s = fmaf(w[4 * l + 2], p.z, s);
            s = fmaf(w[4 * l + 3], p.w, s);
        }
        if (i < n) buffers[cur ^ 1][col][i] = s;
        bar_sync(1, active);
    }
    const float mine = buffers[cur][col][i];
    if (i < n && j < m) out[(int64_t)i * m + j] = mine;
    if (spread) {
        // a maximum is the same in any order, and of numbers that are not negative it is that of their bits (NaN never wins)
        float far = i < n && j < m ? fmaxf(0.f, fabsf(mine - buffers[cur][col][reader])) : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o /= 2) far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, o));
        if (tid % 32 == 0) atomicMax(&worst, __float_as_int(far));
        bar_sync(1, active);
        if (tid == 0) atomicMax(spread, worst);
    }
}

// The rounds alone, for more machines: W in shared memory too.  Rows of W and columns of the messages are read 16 bytes at a
// time, their strides odd multiples of 16 bytes so that the rows a warp reads together fall into different banks.
constexpr int kGossipMaxMachines = 128;               // W in 66 KB of shared memory
__host__ __device__ constexpr int gossip_stride(int n) { return (((n + 3) / 4) | 1) * 4; }
__global__ void gossip_rounds_kernel(const float *W, const float *in, int n, int m, int rounds, float *out) {
    grid_trigger();
    grid_wait();
    extern __shared__ __align__(16) float gossip_smem[];
    const int ld = gossip_stride(n), n4 = (n + 3) / 4;
    float *const weights = gossip_smem, *cur = weights + n * ld, *nxt = cur + kGossipCols * ld;    // W by rows, messages by columns
    const int tid = threadIdx.x, threads = blockDim.x, step = threads / kGossipCols;
    const int col = tid % kGossipCols, first = tid / kGossipCols, j = blockIdx.x * kGossipCols + col;
    for (int i = tid / 32; i < n; i += threads / 32)
        for (int l = tid % 32; l < ld; l += 32) weights[i * ld + l] = l < n ? W[(int64_t)i * n + l] : 0.f;
    for (int i = first; i < ld; i += step) {
        cur[col * ld + i] = i < n && j < m ? __ldcg(in + (int64_t)i * m + j) : 0.f;
        nxt[col * ld + i] = 0.f;
    }
    __syncthreads();
    for (int r = 0; r < rounds; ++r) {
        const float4 *const column = reinterpret_cast<const float4 *>(cur + col * ld);
        for (int i = first; i < n; i += step) {
            const float4 *const row = reinterpret_cast<const float4 *>(weights + i * ld);
            float s = 0.f;
#pragma unroll 4
            for (int l = 0; l < n4; ++l) {
                const float4 w = row[l], p = column[l];
                s = fmaf(w.x, p.x, s);
                s = fmaf(w.y, p.y, s);
                s = fmaf(w.z, p.z, s);
                s = fmaf(w.w, p.w, s);
            }
            nxt[col * ld + i] = s;
        }
        __syncthreads();
        float *const swap = cur;
        cur = nxt;
        nxt = swap;
    }
    if (j < m)
        for (int i = first; i < n; i += step) out[(int64_t)i * m + j] = cur[col * ld + i];
}

// spread[0] = max over machines i and vectors j of |P[i][j] - P[reader][j]| (a maximum: order-free).
__global__ void __launch_bounds__(kSpreadThreads)
consensus_spread_kernel(const float *P, int n, int m, int reader, float *spread) {
    grid_trigger();
    grid_wait();
    __shared__ float part[kSpreadThreads / 32];
    const float *const own = P + (int64_t)reader * m;
    float worst = 0.f;
    // unit = 32 columns of one machine
    const int groups = (m + 31) / 32, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int64_t u = warp; u < (int64_t)groups * n; u += kSpreadThreads / 32) {
        const int i = (int)(u / groups), j = (int)(u % groups) * 32 + lane;
        if (j < m) worst = fmaxf(worst, fabsf(__ldcg(P + (int64_t)i * m + j) - __ldcg(own + j)));
    }
#pragma unroll
    for (int o = 16; o > 0; o /= 2) worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    if (lane == 0) part[warp] = worst;
    __syncthreads();
    if (warp != 0) return;
    worst = part[lane];
#pragma unroll
    for (int o = 16; o > 0; o /= 2) worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    if (lane == 0) *spread = worst;
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

bool gossip_step_applies(int32_t n) { return n <= 64; }
// A CTA finishes the messages of its columns alone, with few threads against the machines where there are more than 32 (us of a
// step, in a launch of their own -> here: 16 machines, d = 2000, m = 64: 25.7 -> 24.2; 32, d = 8192, m = 128: 48.1 -> 47.2; but 40,
// d = 20000, m = 1000: 144.8 -> 148.8; 64, d = 4096, m = 256: 63.1 -> 69.2), and only while a thread adds up few partial sums.
bool gossip_joins(int32_t n, int chunks) {
    const int tasks = n * kGossipCols * kFinishSlices, threads = gossip_threads(n);
    return n <= 32 && (tasks + threads - 1) / threads * ((chunks + kFinishSlices - 1) / kFinishSlices) <= 48;
}

cudaError_t launch_gossip_step(const float *W, const float *partial, int chunks, const float *P, int32_t n, int32_t m, int32_t rounds,
                               float *out, int32_t reader, float *spread, cudaStream_t stream) {
    const int entries = (n + 3) / 4 * 4 * kGossipCols;
    const int most = gossip_threads(n), threads = partial ? (entries * kFinishSlices < most ? entries * kFinishSlices : most) : entries;
    auto go = [&](auto kernel) {
        return launch_chained(true, kernel, dim3((m + kGossipCols - 1) / kGossipCols), dim3(threads), 0, stream, W, partial, chunks, P, n, m, rounds,
                              out, reader, reinterpret_cast<int *>(spread));
    };
    return n <= 16 ? go(gossip_step_kernel<16>) : n <= 32 ? go(gossip_step_kernel<32>) : go(gossip_step_kernel<64>);
}

cudaError_t launch_gossip_rounds(const float *W, float *P, int32_t n, int32_t m, int32_t rounds, float *scratch, float **result,
                                 cudaStream_t stream) {
    *result = P;
    if (rounds <= 0) return cudaSuccess;
    if (n <= kGossipMaxMachines) {
        const size_t smem = ((size_t)n + 2 * kGossipCols) * gossip_stride(n) * sizeof(float);
        const int rows = n <= 4 ? 4 : n < 64 ? (n + 3) / 4 * 4 : 64;           // whole warps
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
    return launch_chained(true, consensus_spread_kernel, dim3(1), dim3(kSpreadThreads), 0, stream, P, n, m, reader, spread);
}

}  // namespace core
