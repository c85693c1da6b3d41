// A whole round of a short vector in one launch: projection, aggregation and reconstruction by one thread-block cluster.
//
// The CTAs of the cluster share out the blocks of the vector.  Each makes the Gaussians of its blocks once, into shared
// memory (nothing of that needs the gradients, so it runs while the kernel before this one drains), multiplies them with its
// part of the gradients, sends its share of the messages to the shared memory of all the others, adds the shares up in the
// order of the CTAs, and reconstructs its blocks from the Gaussians it still has.  Compared with a projection and a
// reconstruction as launches of their own, that saves one hand-over between kernels, the partial sums' way through L2, and half of
// the Gaussians.
// Several machines' messages are formed apart, in the order of the separate kernels (core_project.cu, core_finish.cu): they are the same
// numbers, and so are those of a projection or a reconstruction alone, which are below.
//
// What bounds it: latency.  One hand-over from the previous kernel, one round trip to L2 for the gradients, two cluster barriers, and a
// few dozen counters per thread.
#include "core_emit.cuh"
#include "core_finish.cuh"
#include "core_internal.h"
#include "core_sync.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

namespace core {

namespace {

constexpr int kShortThreads = 512;
constexpr int kShortCluster = 8;                  // most CTAs
constexpr int kShortVectors = 4096;               // most vectors
constexpr int kShortMachines = 8;                 // most messages kept apart
constexpr int kShortLaneBlocks = 16;              // blocks of a lane from which a vector gets more than one warp
constexpr int kShortChainBlocks = 4;              // most blocks of a lane that are added up in one chain
constexpr int kShortSlices = 64;                  // most ranges of the vectors (reconstruction) a block's sum is cut into

struct ShortArgs {
    const void *G;
    int64_t ldg;
    int64_t d;
    int64_t k_end;             // = d (for emit_block)
    int rows;                  // rows added up where there is one message
    int machines;              // messages
    int aligned;               // rows may be read a block at a time
    float scale;
    int m;
    int per;                   // blocks per CTA
    int stride;                // of the Gaussians' rows (one per vector) in shared memory, in blocks
    int lanes;                 // threads that share a vector's projection: a power of two, whole warps from 32 on
    int columns;               // of several messages: the separate kernel's tiles, whose sums are formed as it forms them:
    int tile;                  // blocks of one,
    int tq, uq;                // lanes that share it out, blocks of a lane's step
    int slices;                // ranges of the vectors in the reconstruction
    float *P;                  // not null: the message (there is one) is all that is wanted
    float *pbar;
    float *out;
    int vec_ok;
    uint32_t t;
    RoundKeys keys;
    ReconstructEpilogue epi;
};

__device__ __forceinline__ float4 load_block(const float *row, int64_t k, int64_t d, bool whole) {
    if (whole && k + 4 <= d) return __ldcg(reinterpret_cast<const float4 *>(row + k));
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = k + e < d ? __ldcg(row + k + e) : 0.f;
    return make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ float4 load_block(const __nv_bfloat16 *row, int64_t k, int64_t d, bool whole) {
    if (whole && k + 4 <= d) {                     // a bf16 is the upper half of an fp32
        const uint2 h = __ldcg(reinterpret_cast<const uint2 *>(row + k));
        return make_float4(__uint_as_float(h.x << 16), __uint_as_float(h.x & 0xFFFF0000u), __uint_as_float(h.y << 16),
                           __uint_as_float(h.y & 0xFFFF0000u));
    }
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        v[e] = k + e < d ? __uint_as_float((uint32_t)__ldcg(reinterpret_cast<const unsigned short *>(row) + k + e) << 16) : 0.f;
    return make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void add_block(float4 &s, float4 v) { s = make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w); }

// Blocks of a reconstruction in which the vectors are cut into ranges added up in ascending order, whichever kernel does it.
__device__ __forceinline__ int slice_end(int m, int slice, int slices) { return m * (slice + 1) / slices; }

// The sum of a block's ranges, places[r * stride] for r < ranges (a power of two), in the first `blocks` threads, each a block's.  More than
// eight ranges, up to 64: eight at a time by as many threads first, so that none adds up more than eight in a row.
__device__ __forceinline__ float4 join_ranges(float4 *places, int stride, int ranges, int blocks, int tid) {
    if (ranges > 8) {
        const int group = tid / stride, q = tid - group * stride;
        if (8 * group < ranges && q < blocks) {
            float4 *const first = places + 8 * group * stride + q;
            float4 v[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = first[r * stride];
#pragma unroll
            for (int r = 1; r < 8; ++r) add_block(v[0], v[r]);
            *first = v[0];
        }
        __syncthreads();
        stride *= 8;
        ranges /= 8;
    }
    if (tid >= blocks) return make_float4(0.f, 0.f, 0.f, 0.f);
    float4 s = places[tid];
#pragma unroll 8
    for (int r = 1; r < ranges; ++r) add_block(s, places[r * stride + tid]);
    return s;
}

// The reconstruction alone: the same values and sums, on as many CTAs as there are blocks for, without a cluster.  With parts it
// finishes the message itself, as launch_finish_aggregate does.
__global__ void __launch_bounds__(kShortThreads)
short_reconstruct_kernel(const __grid_constant__ ShortArgs a, const MessageParts parts) {
    grid_trigger();
    extern __shared__ __align__(16) unsigned char smem[];
    uint4 *const table = reinterpret_cast<uint4 *>(smem);                     // {vectors' half of Philox, message}
    float4 *const scratch = reinterpret_cast<float4 *>(table + a.m);          // [thread]
    float *const sums = reinterpret_cast<float *>(scratch + blockDim.x);      // [slice of the columns][machine][vector]
    const int tid = threadIdx.x, threads = blockDim.x, nq = (int)((a.d + 3) >> 2), q0 = (int)blockIdx.x * a.per, mine = min(a.per, nq - q0);
    const int slice = tid / a.per, q = tid - slice * a.per;
    const QPart qp = philox_qpart((uint32_t)(q0 + q), a.t, a.keys);
    for (int j = tid; j < a.m; j += threads) {
        const JPart jp = philox_jpart((uint32_t)j, 0u, a.keys);
        table[j] = make_uint4(jp.x0, jp.x2, jp.w3, 0u);
    }
    grid_wait();
    if (parts.partial) {
        const int entries = parts.n * a.m;
        const bool few = parts.chunks <= kFinishSlices;                       // a column per slice at most: the same sums without them
        if (few)
            for (int e = tid; e < entries; e += threads) sums[e] = sum_strided<8>(parts.partial + e, parts.chunks, entries);
        else
            for (int e = tid; e < entries * kFinishSlices; e += threads)
                sums[e] = finish_slice<8>(parts.partial, parts.chunks, entries, e % entries, e / entries);
        __syncthreads();
        for (int j = tid; j < a.m; j += threads) {
            float sum = 0.f;
            for (int i = 0; i < parts.n; ++i) sum += few ? sums[i * a.m + j] : finish_join(sums + i * a.m + j, entries);
            sum /= (float)parts.n;
            table[j].w = __float_as_uint(sum);
            if (blockIdx.x == 0) a.pbar[j] = sum;
        }
    } else {
        for (int j = tid; j < a.m; j += 4 * threads) {                        // four loads in flight
            float p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = j + i * threads < a.m ? __ldcg(a.pbar + j + i * threads) : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (j + i * threads < a.m) table[j + i * threads].w = __float_as_uint(p[i]);
        }
    }
    __syncthreads();
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (q < mine && slice < a.slices) {
        int j = slice_end(a.m, slice - 1, a.slices);
        const int end = slice_end(a.m, slice, a.slices);
        auto add = [&](auto count) {
            constexpr int N = decltype(count)::value;
            uint4 w[N];
            float p[N];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const uint4 e = table[j + i];
                JPart jp;
                jp.x0 = e.x;
                jp.x2 = e.y;
                jp.w3 = e.z;
                p[i] = __uint_as_float(e.w);
                w[i] = philox_combine(jp, qp, a.keys);
            }
            float4 v[N];
            box_muller4xN<N>(w, v);
#pragma unroll
            for (int i = 0; i < N; ++i) s = make_float4(fmaf(p[i], v[i].x, s.x), fmaf(p[i], v[i].y, s.y), fmaf(p[i], v[i].z, s.z), fmaf(p[i], v[i].w, s.w));
            j += N;
        };
        while (j + 4 <= end) add(std::integral_constant<int, 4>{});
        if (j + 2 < end) add(std::integral_constant<int, 3>{});              // (one by one they would wait for each other)
        else if (j + 1 < end) add(std::integral_constant<int, 2>{});
        else if (j < end) add(std::integral_constant<int, 1>{});
    }
    scratch[tid] = s;
    __syncthreads();
    s = join_ranges(scratch, a.per, a.slices, mine, tid);
    if (tid < mine) {
        const float inv_m = 1.0f / (float)a.m;
        emit_block(a, (uint64_t)(q0 + tid), 0, make_float4(s.x * inv_m, s.y * inv_m, s.z * inv_m, s.w * inv_m));
    }
}

// APART: several messages of a row each, otherwise one, of the sum of the rows.  MANY: more than eight ranges of the vectors (the code that
// joins those, in a kernel that never has them: round of four machines, d = 4096, m = 16: 4.99 -> 5.17 us).
template <typename GT, bool APART, bool MANY>
__global__ void __launch_bounds__(kShortThreads, 1)
short_round_kernel(const __grid_constant__ ShortArgs a) {
    grid_trigger();
    extern __shared__ __align__(16) unsigned char smem[];
    const int per = a.per, m = a.m, tid = threadIdx.x;
    const int machines = APART ? a.machines : 1, entries = machines * m;
    float4 *const z = reinterpret_cast<float4 *>(smem);                       // [vector][block]
    float4 *const g = z + m * a.stride;                                       // [machine][block]
    float4 *const scratch = g + machines * per;                               // [thread]
    uint4 *const vectors = reinterpret_cast<uint4 *>(scratch + kShortThreads);      // the vectors' half of Philox
    float *const inbox = reinterpret_cast<float *>(vectors + m);              // [CTA, or column][machine][vector]
    float *const pbar = inbox + (APART ? a.columns : gridDim.x) * entries;    // [vector]
    float *const sums = pbar + m;                                             // [slice of the columns][machine][vector]
    const uint32_t rank = blockIdx.x, ranks = gridDim.x;                      // one cluster
    const int q0 = (int)rank * per, nq = (int)((a.d + 3) >> 2), mine = max(min(per, nq - q0), 0);
    cluster_arrive();                                                         // this CTA has started

    for (int j = tid; j < m; j += kShortThreads) {
        const JPart jp = philox_jpart((uint32_t)j, 0u, a.keys);
        vectors[j] = make_uint4(jp.x0, jp.x2, jp.w3, 0u);
    }
    __syncthreads();
    {
        // threads of a warp along the blocks, each with a block of its own and every `step`-th vector
        const int step = max(kShortThreads / max(mine, 1), 1);
        for (int q = tid % max(mine, 1); q < mine; q += kShortThreads) {
            const QPart qp = philox_qpart((uint32_t)(q0 + q), a.t, a.keys);
            int j = tid / max(mine, 1);
            if (j >= step) break;
            auto word = [&](int v) {
                const uint4 e = vectors[v];
                JPart jp;
                jp.x0 = e.x;
                jp.x2 = e.y;
                jp.w3 = e.z;
                return philox_combine(jp, qp, a.keys);
            };
            auto make = [&](auto count) {
                constexpr int N = decltype(count)::value;
                uint4 w[N];
#pragma unroll
                for (int s = 0; s < N; ++s) w[s] = word(j + s * step);
                float4 v[N];
                box_muller4xN<N>(w, v);
#pragma unroll
                for (int s = 0; s < N; ++s) z[(j + s * step) * a.stride + q] = v[s];
                j += N * step;
            };
            while (j + 3 * step < m) make(std::integral_constant<int, 4>{});
            if (j + 2 * step < m) make(std::integral_constant<int, 3>{});
            else if (j + step < m) make(std::integral_constant<int, 2>{});
            else if (j < m) make(std::integral_constant<int, 1>{});
        }
    }
    grid_wait();

    // this CTA's part of the gradients
    const GT *const G = static_cast<const GT *>(a.G);
    if (!APART && a.rows > 1) {
        // the rows in as many ranges as there are threads for, added up in the order of the ranges
        const int ranges = mine > 0 ? min(kShortThreads / min(mine, kShortThreads), (a.rows + 7) / 8) : 1;
        for (int qb = 0; qb < mine; qb += kShortThreads) {
            const int here = min(mine - qb, kShortThreads), q = tid % here, range = tid / here;
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
            if (range < ranges) {
                const int64_t k = (int64_t)(q0 + qb + q) << 2;
                const int end = a.rows * (range + 1) / ranges;
                for (int r = a.rows * range / ranges; r < end; r += 8) {          // eight loads in flight, also of the last ones
                    float4 v[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        v[i] = r + i < end ? load_block(G + (int64_t)(r + i) * a.ldg, k, a.d, a.aligned) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < 8; ++i) add_block(s, v[i]);
                }
            }
            if (ranges > 1) {
                scratch[tid] = s;
                __syncthreads();
                if (range == 0) {
#pragma unroll 8
                    for (int r = 1; r < ranges; ++r) add_block(s, scratch[r * here + q]);
                }
            }
            if (range == 0) g[qb + q] = make_float4(s.x * a.scale, s.y * a.scale, s.z * a.scale, s.w * a.scale);
            __syncthreads();
        }
    } else {
        for (int e = tid; e < machines * mine; e += 4 * kShortThreads) {              // four loads in flight
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = (e + u * kShortThreads) / mine, q = (e + u * kShortThreads) % mine;
                v[u] = i < machines ? load_block(G + (int64_t)i * a.ldg, (int64_t)(q0 + q) << 2, a.d, a.aligned) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = (e + u * kShortThreads) / mine, q = (e + u * kShortThreads) % mine;
                const float scale = APART ? 1.f : a.scale;
                if (i < machines) g[i * per + q] = make_float4(v[u].x * scale, v[u].y * scale, v[u].z * scale, v[u].w * scale);
            }
        }
    }
    __syncthreads();

    // its share of every message, to all CTAs
    cluster_wait();                                                           // they have all started
    if constexpr (APART) {
        // A column's share of a message by one thread, in the order in which the separate kernel adds it up (lane by lane of those that
        // share its tile out there), so that it is the same number.
        const int column0 = (int)rank * (per / a.tile), mine_columns = (mine + a.tile - 1) / a.tile;
        for (int task = tid; task < mine_columns * entries; task += kShortThreads) {
            const int column = task / entries, e = task % entries, q_base = column * a.tile, blocks = min(a.tile, mine - q_base);
            const float4 *const zz = z + (e % m) * a.stride + q_base, *const gg = g + (e / m) * per + q_base;
            float sum = 0.f;
            constexpr int L = 8;                                              // lanes side by side
            for (int l0 = 0; l0 < a.tq; l0 += L) {
                float p[L] = {};
                for (int first = l0 * a.uq; first < blocks; first += a.tq * a.uq)
                    for (int u = 0; u < a.uq; ++u) {
                        float4 v[L], b[L];
#pragma unroll
                        for (int i = 0; i < L; ++i) {
                            const int q = first + i * a.uq + u;
                            const bool there = l0 + i < a.tq && q < blocks;
                            v[i] = zz[there ? q : 0];
                            b[i] = there ? gg[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                        for (int i = 0; i < L; ++i) {
                            p[i] = fmaf(b[i].x, v[i].x, p[i]);
                            p[i] = fmaf(b[i].y, v[i].y, p[i]);
                            p[i] = fmaf(b[i].z, v[i].z, p[i]);
                            p[i] = fmaf(b[i].w, v[i].w, p[i]);
                        }
                    }
#pragma unroll
                for (int i = 0; i < L; ++i) sum += p[i];
            }
            for (uint32_t r = 0; r < ranks; ++r) store_remote(inbox + (column0 + column) * entries + e, r, sum);
        }
    } else {
        // Up to four blocks of a lane in one chain of up to 16 additions, more in four sums, whose chains are as long as the lane has blocks
        // (rms error of a message, of the gradient's norm, m = 64, d = 2900, twelve blocks: one chain 1.8e-7, four sums 1.5e-7).
        const bool chain = per <= kShortChainBlocks * a.lanes;
        const auto dot = [&](int j, int sub) {
            if (chain) {
                float p = 0.f;
                if (j < m)
                    for (int q = sub; q < mine; q += a.lanes) {
                        const float4 v = z[j * a.stride + q], b = g[q];
                        p = fmaf(b.x, v.x, p);
                        p = fmaf(b.y, v.y, p);
                        p = fmaf(b.z, v.z, p);
                        p = fmaf(b.w, v.w, p);
                    }
                return p;
            }
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j < m)
                for (int q = sub; q < mine; q += a.lanes) {
                    const float4 v = z[j * a.stride + q], b = g[q];
                    s = make_float4(fmaf(b.x, v.x, s.x), fmaf(b.y, v.y, s.y), fmaf(b.z, v.z, s.z), fmaf(b.w, v.w, s.w));
                }
            return (s.x + s.y) + (s.z + s.w);
        };
        if (a.lanes <= 32) {
            for (int j0 = 0; j0 < m; j0 += kShortThreads / a.lanes) {
                const int sub = tid & (a.lanes - 1), j = j0 + tid / a.lanes;
                float p = dot(j, sub);
                for (int o = a.lanes / 2; o > 0; o /= 2) p += __shfl_xor_sync(0xffffffffu, p, o);
                if (j < m)
                    for (uint32_t r = sub; r < ranks; r += a.lanes) store_remote(inbox + rank * m + j, r, p);
            }
        } else {                                                              // several warps per vector: all vectors are here at once
            const int sub = tid & (a.lanes - 1), j = tid / a.lanes, warps = a.lanes / 32;
            float p = dot(j, sub);
            for (int o = 16; o > 0; o /= 2) p += __shfl_xor_sync(0xffffffffu, p, o);
            float *const part = reinterpret_cast<float *>(scratch);
            if (tid % 32 == 0) part[tid / 32] = p;
            __syncthreads();
            if (j < m && sub < (int)ranks) {
                p = part[j * warps];
                for (int w = 1; w < warps; ++w) p += part[j * warps + w];
                store_remote(inbox + rank * m + j, sub, p);
            }
        }
    }
    cluster_arrive();
    cluster_wait();
    if constexpr (APART) {
        // the columns as the finishing kernels add them up, then the mean over the machines (up to eight columns, a slice each at most, in the
        // same way: a second way in the kernel cost all rounds more, four machines, d = 4096, m = 16: 5.17 -> 5.27 us, d = 700: 4.17 -> 4.34)
        for (int e = tid; e < entries * kFinishSlices; e += kShortThreads) {
            const int entry = e % entries, slice = e / entries, end = a.columns * (slice + 1) / kFinishSlices;
            float s = 0.f;
#pragma unroll 4
            for (int c = a.columns * slice / kFinishSlices; c < end; ++c) s += inbox[c * entries + entry];
            sums[e] = s;
        }
        __syncthreads();
    }
    for (int j = tid; j < m; j += kShortThreads) {
        float sum = 0.f;
        if constexpr (APART) {
            for (int i = 0; i < machines; ++i) sum += finish_join(sums + i * m + j, entries);
            sum /= (float)machines;
        } else {
#pragma unroll 8
            for (uint32_t r = 0; r < ranks; ++r) sum += inbox[r * m + j];
        }
        if (a.P) {
            if (rank == 0) a.P[j] = sum;                                      // a single message
        } else {
            pbar[j] = sum;
            if (rank == 0) a.pbar[j] = sum;
        }
    }
    if (a.P) return;
    __syncthreads();

    // the blocks of this CTA, `pass` at a time, the vectors of each in ranges that are added up in ascending order
    const int pass = min(per, kShortThreads / a.slices);
    for (int qb = 0; qb < mine; qb += pass) {
        const int here = min(mine - qb, pass), slices = a.slices;
        const int q = tid % pass, slice = tid / pass;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (slice < slices && q < here) {
            const int end = slice_end(m, slice, slices);
#pragma unroll 4
            for (int j = slice_end(m, slice - 1, slices); j < end; ++j) {
                const float4 v = z[j * a.stride + qb + q];
                const float p = pbar[j];
                s = make_float4(fmaf(p, v.x, s.x), fmaf(p, v.y, s.y), fmaf(p, v.z, s.z), fmaf(p, v.w, s.w));
            }
            scratch[tid] = s;
        }
        __syncthreads();
        if constexpr (MANY) s = join_ranges(scratch, pass, slices, here, tid);
        if (tid < here) {
            if constexpr (!MANY) {
#pragma unroll 8
                for (int r = 1; r < slices; ++r) add_block(s, scratch[r * pass + q]);
            }
            const float inv_m = 1.0f / (float)m;
            emit_block(a, (uint64_t)(q0 + qb + q), 0, make_float4(s.x * inv_m, s.y * inv_m, s.z * inv_m, s.w * inv_m));
        }
        __syncthreads();
    }
}

}  // namespace

namespace {
bool g_off = false;
}
void short_kernels_set(bool on) { g_off = !on; }
bool short_kernels_off() { return g_off; }

// Where the one launch applies.  Most counters (m times the blocks) for one message, two to four, five to eight; us, a round by separate
// kernels -> by one: one machine, m = 64, 9600 counters: 6.8 -> 3.4, m = 8, 48000: 6.7 -> 5.4, m = 16, 65536: 6.0 -> 6.3; four machines, m = 24,
// 12000: 6.5 -> 5.0, m = 24, 36000: 7.9 -> 8.3; eight machines, m = 8, 4000: 5.9 -> 4.4.  Few columns for many vectors (four machines, d = 54,
// m = 256: 7.1 -> 17.2 by one CTA) keep the separate kernels.
constexpr int kShortCounters[3] = {48 << 10, 24 << 10, 8 << 10};
// Few vectors leave a thread more blocks than vectors, one after the other: up to 2560 blocks per CTA (m = 1: d = 192 670: 11.8 -> 12.6, d = 88 472:
// 8.0 -> 7.6).
// Several messages of few vectors: the columns of a warp's threads lie in the same banks, and few threads have a column. So
// only columns of the small tiles, fewer than 4096 blocks of all machines per CTA, and no more than 13 312 sums of a vector and a machine's block (us: two
// machines, m = 1, d = 44 234: 7.0 -> 13.2; eight, m = 1, d = 32 111: 8.3 -> 16.6; eight, m = 2, d = 16 054: 7.5 -> 9.9; four, m = 37, d = 2599:
// 7.5 -> 7.6; but three, m = 3, d = 14 744: 7.8 -> 5.8).
constexpr int kShortApartBlocks = 4096, kShortApartSums = 13 << 10;
// Partial gradients take longer to add up on eight SMs than on all, the more the longer a CTA's part is, and what follows is in
// series with it: per block of a CTA two units for a row, four for a vector and forty. us, steps by separate kernels -> by one:
// 148 rows, d = 2561, m = 65: 16.0 -> 18.9 (48 276 units); 26 rows, d = 18 174, m = 2: 15.7 -> 17.6 (56 800); 80 rows, d = 5000, m = 24: 11.9 -> 12.9
// (46 472); but 8 rows, d = 16 000, m = 8: 13.9 -> 12.9 (44 000); 148 rows, d = 3500, m = 8: 16.2 -> 12.3 (40 480).
constexpr int kShortRowUnits = 44000;
constexpr int kShortBlocks = 2560;
ShortPlan make_short_plan(int32_t machines, int32_t rows, int32_t m, int64_t d, int sm_count) {
    ShortPlan p{};
    const int64_t nq = (d + 3) >> 2;
    if (machines > kShortMachines || m > kShortVectors || nq * m > kShortCounters[machines == 1 ? 0 : machines <= 4 ? 1 : 2]) return p;
    const bool apart = machines > 1;
    int64_t units = nq;                                        // that the CTAs share out
    p.tile = 1;
    if (apart) {
        const ProjectPlan separate = make_project_plan(machines, m, d, 0, sm_count);
        if (separate.tc || separate.tiles > separate.grid_x) return p;
        p.tile = separate.tile_q;
        p.tq = separate.tq;
        p.uq = separate.uq;
        units = separate.tiles;
    }
    if (apart && nq * m > 512 * units && units < kShortCluster) return p;       // too few columns to share out
    int ctas = 1;
    while (ctas < kShortCluster && nq * m > (int64_t)256 * ctas && ctas < units) ctas *= 2;
    p.columns = (int)units;
    p.per = (int)((units + ctas - 1) / ctas) * p.tile;
    if (apart && (p.tile > 32 || (int64_t)machines * p.per >= kShortApartBlocks || (int64_t)machines * p.per * m > kShortApartSums)) return p;
    p.stride = p.per | 1;
    p.lanes = 1;
    // up to a warp per vector, several warps where that leaves a lane more than sixteen blocks in a row (m = 3, d = 64 000: 63, and the error of the
    // message, rms, 3.3e-7 of the gradient's norm, where the separate kernels' is 3.0e-7 and this 1.7e-7)
    while ((p.lanes < 32 ? p.lanes : kShortLaneBlocks * p.lanes) < p.per && 2 * p.lanes * m <= kShortThreads) p.lanes *= 2;
    p.slices = 1;
    while (p.slices < kShortSlices && 6 * p.slices <= m) p.slices *= 2;      // three vectors and more in each
    // per CTA: the Gaussians, its part of the rows, a 16-byte place per thread, the vectors' half of Philox; the shares of the messages, the
    // combined message, the columns' slices
    const size_t entries = (size_t)machines * m;
    p.smem = ((size_t)m * p.stride + (size_t)machines * p.per + kShortThreads + m) * 16 +
             ((apart ? p.columns + kFinishSlices : ctas) * entries + m) * 4;
    if (rows > 1 && (2 * (int64_t)rows + 4 * m + 40) * p.per > kShortRowUnits) return p;
    if (p.smem <= 200 * 1024 && p.per <= kShortBlocks) p.ctas = ctas;
    return p;
}

// At most a CTA per SM, and four warps each: a step's next kernel wants the other SMs early (17 machines, d = 313, m = 9: a warp
// on ten SMs made a step of 26.7 us one of 27.8).  A thread per block and range, and threads for the table of the vectors.
// With parts every CTA finishes the whole message: half as many CTAs, of eight warps, and a thread per sum, as far as 512 go, since a
// thread's sums wait for L2 one after the other (us, rounds of three machines, m = 200, d = 219: 17.0 -> 6.9; five, m = 100, d = 141:
// 15.2 -> 6.4; accelerated steps by separate kernels, with the 128 threads and twice as many CTAs: 40 rows, d = 16000, m = 8: 14.4 instead of 15.8).
ShortGrid make_short_grid(const ShortPlan &plan, int32_t m, int64_t d, int sm_count, const MessageParts *parts) {
    const int nq = (int)((d + 3) >> 2), most = kShortThreads / plan.slices, least = (parts ? 256 : 128) / plan.slices;
    const int sums = parts ? parts->n * m * (parts->chunks > kFinishSlices ? kFinishSlices : 1) : 0;
    ShortGrid g;
    g.per = std::clamp((nq + sm_count - 1) / sm_count, least, most);
    g.threads = (std::max({g.per * plan.slices, std::min(m / 2, kShortThreads), std::min(sums, kShortThreads)}) + 31) / 32 * 32;
    g.ctas = (nq + g.per - 1) / g.per;
    return g;
}

static ShortArgs short_args(const ShortPlan &plan, const RoundKeys &keys, uint32_t t, int64_t d, int32_t m, float *pbar, float *out,
                            const ReconstructEpilogue *epilogue) {
    ShortArgs a{};
    a.d = a.k_end = d;
    a.m = m;
    a.per = plan.per;
    a.stride = plan.stride;
    a.lanes = plan.lanes;
    a.columns = plan.columns;
    a.tile = plan.tile;
    a.tq = plan.tq;
    a.uq = plan.uq;
    a.slices = plan.slices;
    a.pbar = pbar;
    a.out = out;
    uintptr_t align = reinterpret_cast<uintptr_t>(out);
    if (epilogue && epilogue->base) {
        a.epi = *epilogue;
        align |= reinterpret_cast<uintptr_t>(epilogue->base);
        if (epilogue->shift_dst) align |= reinterpret_cast<uintptr_t>(epilogue->shift_src) | reinterpret_cast<uintptr_t>(epilogue->shift_dst);
    }
    a.vec_ok = align % 16 == 0 ? 1 : 0;
    a.t = t;
    a.keys = keys;
    return a;
}

cudaError_t launch_short_round(const ShortPlan &plan, const RoundKeys &keys, uint32_t t, const void *G, int dtype, int32_t rows,
                               int32_t machines, int64_t ldg, float scale, int64_t d, int32_t m, float *P, float *pbar, float *out,
                               const ReconstructEpilogue *epilogue, cudaStream_t stream) {
    ShortArgs a = short_args(plan, keys, t, d, m, pbar, out, epilogue);
    a.G = G;
    a.ldg = ldg;
    a.rows = rows;
    a.machines = machines;
    a.aligned = reinterpret_cast<uintptr_t>(G) % (dtype == 1 ? 8 : 16) == 0 && ldg % 4 == 0;
    a.scale = scale;
    a.P = P;
    auto go = [&](auto kernel) {
        if (cudaError_t e = allow_shared(reinterpret_cast<const void *>(kernel), plan.smem)) return e;
        const ChainedLaunch launch(true, dim3((unsigned)plan.ctas), dim3(kShortThreads), plan.smem, stream, plan.ctas);
        return cudaLaunchKernelEx(&launch.cfg, kernel, a);
    };
    auto pick = [&](auto gt, auto many) {
        using GT = decltype(gt);
        return machines == 1 ? go(short_round_kernel<GT, false, many.value>) : go(short_round_kernel<GT, true, many.value>);
    };
    if (dtype == 1) return plan.slices > 8 ? pick(__nv_bfloat16{}, std::true_type{}) : pick(__nv_bfloat16{}, std::false_type{});
    return plan.slices > 8 ? pick(0.f, std::true_type{}) : pick(0.f, std::false_type{});
}

cudaError_t launch_short_reconstruct(const ShortPlan &plan, const RoundKeys &keys, uint32_t t, float *pbar, int64_t d, int32_t m, float *out,
                                     int sm_count, const ReconstructEpilogue *epilogue, const MessageParts *parts, cudaStream_t stream) {
    ShortArgs a = short_args(plan, keys, t, d, m, pbar, out, epilogue);
    const ShortGrid grid = make_short_grid(plan, m, d, sm_count, parts);
    a.per = grid.per;
    const MessageParts join = parts ? *parts : MessageParts{};
    const size_t smem = ((size_t)m + grid.threads) * 16 + (parts ? (size_t)kFinishSlices * parts->n * m * 4 : 0);
    return launch_chained(true, short_reconstruct_kernel, dim3((unsigned)grid.ctas), dim3(grid.threads), smem, stream, a, join);
}

}  // namespace core
