// Projection of one combined gradient row: p_j = <scale * sum_r G_r, xi_j>, j < m.
//
// Used for a single machine, for the least-squares steps (the rows are the partial gradients of the row
// ranges) and for rounds whose per-machine messages nobody asks for: the mean message is linear in the
// gradients, pbar_j = (1/n) sum_i <g_i, xi_j> = <(1/n) sum_i g_i, xi_j>, so adding the gradients while they
// are staged (n d additions) replaces the n d m multiply-adds of n separate messages by d m.
//
// What bounds it: the generator (see core_rng.cuh), like the other round kernels; with few vectors and many
// rows, the reading of G.  A CTA has generating warps and a few staging warps.  The staging warps read the
// rows of the next tile 16 bytes at a time (eight loads in flight per thread), add them up and store the
// sum to one of two shared-memory tiles, next to the block-dependent half of Philox; rows that
// do not start on a 16-byte boundary are read in aligned vectors all the same, summed per alignment class
// and shifted into place with warp shuffles.  Where rows are many against the vectors, every warp stages and
// then generates, and the other CTA of the SM fills the gap.  The generating threads hold four
// vectors each and walk the blocks of the tile: thread (jl, ql) of tj x tq, where tj = the number of vector
// quadruples of the CTA row (any number, not a power of two: 100 vectors keep 750 of 768 threads busy).  The
// coordinates of a block are stored as (0, 2, 1, 3), so that one 16-byte read delivers the multiplicands of the
// cosine and of the sine lanes of both pairs as ready register pairs and S (g_c cos + g_s sin) is two packed and two
// scalar instructions per counter.
//
// Three modes.  kRowTurn, wherever there is work for it: angles from the table, one CTA of 24 generating and 4 staging warps
// per SM, d = 2.56e7, m = 256: 4944 us = 1.32e12 Gaussians/s.  kRowShort: angles from the polynomials, two CTAs of 8 and 2
// warps per SM (d = 2.5e7: 5325 us, with the table 4904), for short work.  kRowTogether: the same, all warps stage.  In kRowTurn the registers decide:
// 72 per thread hold the loop only because the sums over tiles live in shared memory and scalar accumulators
// (packed ones need pairs: 5138 us) and 32-bit counts go around it (64-bit tile numbers: 5095); 20 generating warps of 80 registers:
// 5169, 28 of 64: 5144, two counters at a time: 5379.
// The generating warps take tiles over in three groups of eight, each with barriers of its own: with one barrier for all, every warp
// waited for the slowest one at each tile (us, one group -> three: d = 2.5e7, m = 256: 4958 -> 4904; d = 1e6, m = 100:
// 88.7 -> 87.9; eight rows, d = 1e7, the whole round: 3838 -> 3805).
#include "core_internal.h"
#include "core_sync.cuh"

#include <algorithm>

#include <cuda_bf16.h>

#include <climits>

namespace core {

namespace {

constexpr int kRowJT = 4;                        // vectors per generating thread
// Steps that are added up before they meet the sum of all: the longest chain of additions but that one, which has as many links as a CTA's
// tiles have such parts.  A message's rounding error grows with the square root of such a chain: 64 steps made that of rows whose CTAs
// have one long tile a quarter larger (d = 1 000 003, m = 100: rms 1.76e-7 of the row's norm -> 2.31e-7).
constexpr int kRowSumSteps = 32;

// With the table of angles one CTA fills an SM, without it two do.
template <bool TURN>
struct RowCta {
    static constexpr int kCompute = TURN ? 768 : 256;        // generating threads
    static constexpr int kStagers = TURN ? 128 : 64;         // staging threads
    static constexpr int kThreads = kCompute + kStagers;
    static constexpr int kGroups = TURN ? 3 : 1;             // of generating warps that take a tile over by themselves
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kPerSm = TURN ? 1 : 2;
    static constexpr int kTileBlocks = TURN ? 2048 : 1024;   // most blocks of a tile,
    static constexpr int kTileSteps = TURN ? 128 : 64;       // and most steps of a generating thread in one
};

struct RowArgs {
    const void *G;
    int64_t ldg;
    int64_t d;
    int64_t tiles;
    uint64_t q_base;
    float *partial;
    int rows;
    int period;      // rows r and r + period have the same alignment
    int aligned;     // every tile of every row starts on a 16-byte boundary
    float scale;
    int m;
    int tile_q;      // coordinate blocks per tile
    int tj;          // threads across vectors
    int tq;          // threads across blocks: tj * tq generating threads at most
    uint32_t t;
    RoundKeys keys;
};

template <typename GT>
struct RowVec {
    static constexpr int V = 16 / (int)sizeof(GT);          // elements per 16-byte vector
};

__device__ __forceinline__ float row_elem(const float *p) { return __ldcg(p); }
__device__ __forceinline__ float row_elem(const __nv_bfloat16 *p) {
    return __uint_as_float((uint32_t)__ldcg(reinterpret_cast<const unsigned short *>(p)) << 16);
}

__device__ __forceinline__ void row_add(float (&acc)[4], uint4 h) {
    acc[0] += __uint_as_float(h.x);
    acc[1] += __uint_as_float(h.y);
    acc[2] += __uint_as_float(h.z);
    acc[3] += __uint_as_float(h.w);
}
__device__ __forceinline__ void row_add(float (&acc)[8], uint4 h) {      // a bf16 is the upper half of an fp32
    acc[0] += __uint_as_float(h.x << 16);
    acc[1] += __uint_as_float(h.x & 0xFFFF0000u);
    acc[2] += __uint_as_float(h.y << 16);
    acc[3] += __uint_as_float(h.y & 0xFFFF0000u);
    acc[4] += __uint_as_float(h.z << 16);
    acc[5] += __uint_as_float(h.z & 0xFFFF0000u);
    acc[6] += __uint_as_float(h.w << 16);
    acc[7] += __uint_as_float(h.w & 0xFFFF0000u);
}

// acc[u] += rows r0, r0 + period, ... < r1 of the vectors at elements kv + u * stride of their rows.
template <int US, int UR, typename GT, int V>
__device__ __forceinline__ void row_sum(const RowArgs &a, int64_t kv, int64_t stride, int r0, int r1, float (&acc)[US][V]) {
    const GT *G = static_cast<const GT *>(a.G);
    const int step = a.period;
    const int64_t row_stride = (int64_t)step * a.ldg;
    if (kv >= 0 && kv + (US - 1) * stride + V <= a.d) {
        const GT *p = G + (int64_t)r0 * a.ldg + kv;
        for (int r = r0; r < r1; r += UR * step, p += UR * row_stride) {
            uint4 h[US][UR];
#pragma unroll
            for (int i = 0; i < UR; ++i)
#pragma unroll
                for (int u = 0; u < US; ++u)
                    h[u][i] = r + i * step < r1 ? __ldcg(reinterpret_cast<const uint4 *>(p + i * row_stride + u * stride))
                                                : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int i = 0; i < UR; ++i)
#pragma unroll
                for (int u = 0; u < US; ++u) row_add(acc[u], h[u][i]);
        }
        return;
    }
    // some vector of this thread reaches beyond a row's ends: element by element, nothing outside [0, d)
    for (int r = r0; r < r1; r += step) {
        const GT *p = G + (int64_t)r * a.ldg;
#pragma unroll
        for (int u = 0; u < US; ++u)
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const int64_t k = kv + u * stride + e;
                if (k >= 0 && k < a.d) acc[u][e] += row_elem(p + k);
            }
    }
}

// Moves the lanes' vectors (a contiguous run of 32 V elements, continued by lane 31's `ext`) down by W elements.
template <int W, int V>
__device__ __forceinline__ void row_shift(float (&acc)[V], float (&ext)[V], int lane) {
    float in[W];
#pragma unroll
    for (int e = 0; e < W; ++e) {
        const float from_next = __shfl_down_sync(0xffffffffu, acc[e], 1);
        in[e] = lane == 31 ? ext[e] : from_next;
    }
#pragma unroll
    for (int e = 0; e < V; ++e) acc[e] = e + W < V ? acc[e + W] : in[e + W - V];
#pragma unroll
    for (int e = 0; e + W < V; ++e) ext[e] = ext[e + W];
}

// Sum of rows [r0, r1) for the US segments of 32 V coordinates at k, k + 32 V, ...: lane l gets coordinates
// k + 32 V u + V l + e.
template <int US, int UR, bool ALIGNED, typename GT>
__device__ __forceinline__ void row_segments(const RowArgs &a, int64_t k, int r0, int r1, int lane, float (&sum)[US][RowVec<GT>::V]) {
    constexpr int V = RowVec<GT>::V;
#pragma unroll
    for (int u = 0; u < US; ++u)
#pragma unroll
        for (int e = 0; e < V; ++e) sum[u][e] = 0.f;
    if constexpr (ALIGNED) {
        row_sum<US, UR, GT, V>(a, k + V * lane, 32 * V, r0, r1, sum);
    } else {
        for (int c = 0; c < a.period && r0 + c < r1; ++c) {
            // elements between the 16-byte boundary below and coordinate k of the rows of this class
            const uintptr_t at = reinterpret_cast<uintptr_t>(static_cast<const GT *>(a.G) + (int64_t)(r0 + c) * a.ldg + k);
            const int s = (int)((at / sizeof(GT)) & (V - 1));
            if (s == 0) {
                row_sum<US, UR, GT, V>(a, k + V * lane, 32 * V, r0 + c, r1, sum);
                continue;
            }
            float acc[US][V], ext[US][V];
#pragma unroll
            for (int u = 0; u < US; ++u)
#pragma unroll
                for (int e = 0; e < V; ++e) acc[u][e] = ext[u][e] = 0.f;
            row_sum<US, UR, GT, V>(a, k - s + V * lane, 32 * V, r0 + c, r1, acc);
            if (lane == 31) row_sum<US, UR, GT, V>(a, k - s + 32 * V, 32 * V, r0 + c, r1, ext);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < US; ++u) {
                if (s & 1) row_shift<1, V>(acc[u], ext[u], lane);
                if (s & 2) row_shift<2, V>(acc[u], ext[u], lane);
                if constexpr (V == 8)
                    if (s & 4) row_shift<4, V>(acc[u], ext[u], lane);
#pragma unroll
                for (int e = 0; e < V; ++e) sum[u][e] += acc[u][e];
            }
        }
    }
}

// Segments first, first + step, ... of the tile at coordinate k0 (`blocks` of its blocks exist) into `tile`, `stride` float4
// apart per block.
template <int US, int UR, bool ALIGNED, typename GT>
__device__ __forceinline__ void row_stage(int stride, const RowArgs &a, int64_t k0, int blocks, int first, int step, int r0, int r1, int lane,
                                          float4 *tile) {
    constexpr int V = RowVec<GT>::V;
    constexpr int SB = 8 * V;                                // blocks per segment
    const int segments = (blocks + SB - 1) / SB;
    for (int sg = first * US; sg < segments; sg += step * US) {
        float sum[US][V];
        row_segments<US, UR, ALIGNED, GT>(a, k0 + (int64_t)sg * (32 * V), r0, r1, lane, sum);
#pragma unroll
        for (int u = 0; u < US; ++u)
#pragma unroll
            for (int b = 0; b < V / 4; ++b) {
                const int q = (sg + u) * SB + lane * (V / 4) + b;
                if (q < blocks)
                    tile[q * stride] = make_float4(sum[u][4 * b] * a.scale, sum[u][4 * b + 2] * a.scale, sum[u][4 * b + 1] * a.scale,
                                          sum[u][4 * b + 3] * a.scale);
            }
    }
}

// More segments at once where there are few rows to read per segment: about eight loads in flight either way, twelve
// where there are many rows (n = 50, m = 21, d = 1.2e7: 1596 -> 951 us together with eight for unaligned rows).
template <typename GT>
__device__ __forceinline__ void row_stage_any(int stride, const RowArgs &a, int64_t k0, int blocks, int first, int step, int r0, int r1,
                                              int lane, float4 *tile) {
    const int per_class = (r1 - r0 + a.period - 1) / a.period;
    if (a.aligned) {
        if (per_class <= 2) row_stage<RowVec<GT>::V == 4 ? 4 : 2, 2, true, GT>(stride, a, k0, blocks, first, step, r0, r1, lane, tile);
        else if (per_class > 8) row_stage<1, 12, true, GT>(stride, a, k0, blocks, first, step, r0, r1, lane, tile);
        else row_stage<1, 8, true, GT>(stride, a, k0, blocks, first, step, r0, r1, lane, tile);
    } else {
        if (per_class <= 2) row_stage<2, 2, false, GT>(stride, a, k0, blocks, first, step, r0, r1, lane, tile);
        else row_stage<1, 8, false, GT>(stride, a, k0, blocks, first, step, r0, r1, lane, tile);
    }
}

enum RowMode { kRowShort, kRowTogether, kRowTurn };

template <typename GT, RowMode MODE>
__global__ void __launch_bounds__(RowCta<MODE == kRowTurn>::kThreads, RowCta<MODE == kRowTurn>::kPerSm)
project_row_kernel(const __grid_constant__ RowArgs a) {
    constexpr bool TOGETHER = MODE == kRowTogether, TURN = MODE == kRowTurn;
    constexpr int kRowCompute = RowCta<TURN>::kCompute, kRowStagers = RowCta<TURN>::kStagers, kRowThreads = RowCta<TURN>::kThreads,
                  kRowWarps = RowCta<TURN>::kWarps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // two tiles of {coordinates of the combined row, QPart} per block, side by side so that a step addresses both
    // with one pointer (two separate arrays: 5426 against 5276 us at d = 2.5e7, m = 256)
    float4 *const tile0 = reinterpret_cast<float4 *>(smem_raw + (TURN ? kTurnBytes + kRowJT * 4 * RowCta<true>::kCompute : 0));
    const float2 *const turns = reinterpret_cast<const float2 *>(smem_raw);
    float *const totals = reinterpret_cast<float *>(smem_raw + kTurnBytes);
    constexpr int kSegBlocks = 8 * RowVec<GT>::V;
    constexpr int kGroups = RowCta<TURN>::kGroups, kHandOver = kRowCompute / kGroups + kRowStagers;     // threads of a group's barriers
    constexpr int kFull = 1, kEmpty = kFull + 2 * kGroups, kLast = kEmpty + 2 * kGroups;                // barrier ids: + 2 group + stage
    static_assert(kLast < 16, "barriers of a CTA");

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t tile_begin = a.tiles * (int64_t)blockIdx.x / gridDim.x;
    const int64_t tile_end = a.tiles * (int64_t)(blockIdx.x + 1) / gridDim.x;
    const int64_t nq = (a.d + 3) >> 2;
    auto blocks_of = [&](int64_t tile) { return (int)min((int64_t)a.tile_q, nq - tile * a.tile_q); };
    auto fill_table = [&](int64_t tile, float4 *dst, int first, int step) {
        const uint32_t q0 = (uint32_t)(a.q_base + (uint64_t)tile * a.tile_q);
        for (int e = first; e < blocks_of(tile); e += step) {
            const QPart qp = philox_qpart(q0 + (uint32_t)e, a.t, a.keys);
            reinterpret_cast<uint4 *>(dst)[2 * e + 1] = make_uint4(qp.hi_b, qp.lo_b, qp.w3, 0u);
        }
    };

    if constexpr (TURN) fill_turn_table<kRowWarps>(reinterpret_cast<float2 *>(smem_raw), warp, lane);
    const int ql = tid / a.tj, jl = tid - ql * a.tj, jbase = blockIdx.y * a.tj * kRowJT;
    auto first_q = [&] { return a.q_base + (uint64_t)tile_begin * a.tile_q; };
    JPart jp[kRowJT];
    auto make_jp = [&](uint32_t q_hi) {
#pragma unroll
        for (int v = 0; v < kRowJT; ++v) jp[v] = philox_jpart((uint32_t)(jbase + jl + v * a.tj), q_hi, a.keys);
    };
    if (tile_begin < tile_end) fill_table(tile_begin, tile0, tid, kRowThreads);
    grid_wait();

    // the first tile is staged by all warps, nobody having anything else to do yet; a short tile with many rows (the
    // partial gradients of a least-squares step) is cut into row ranges too
    if (tile_begin < tile_end) {
        const int blocks = blocks_of(tile_begin), segments = (blocks + kSegBlocks - 1) / kSegBlocks;
        const int ranges = a.rows >= 2 * kRowWarps ? kRowWarps / segments : 1;
        if (ranges > 1) {
            float4 *const scratch = tile0 + 2 * a.tile_q;    // the second tile's place: it is staged after the barrier below
            const int range = warp / segments;
            const int per = ((a.rows + ranges - 1) / ranges + a.period - 1) / a.period * a.period;
            if (range < ranges)
                row_stage_any<GT>(1, a, 4 * tile_begin * a.tile_q, blocks, warp % segments, segments, min(range * per, a.rows),
                                  min((range + 1) * per, a.rows), lane, scratch + range * blocks);
            __syncthreads();
            for (int q = tid; q < blocks; q += kRowThreads) {
                float4 s = scratch[q];
                for (int r = 1; r < ranges; ++r) {
                    const float4 p = scratch[r * blocks + q];
                    s = make_float4(s.x + p.x, s.y + p.y, s.z + p.z, s.w + p.w);
                }
                tile0[2 * q] = s;
            }
        } else {
            row_stage_any<GT>(2, a, 4 * tile_begin * a.tile_q, blocks, warp, kRowWarps, 0, a.rows, lane, tile0);
        }
    }
    __syncthreads();

    if (warp >= kRowCompute / 32 && !TOGETHER) {
        // staging warps: tile i into stage i & 1 once the generating warps have left it
        for (int64_t tile = tile_begin + 1; tile < tile_end; ++tile) {
            const int i = (int)(tile - tile_begin), st = i & 1;
            if (i >= 2)
                for (int g = 0; g < kGroups; ++g) bar_sync(kEmpty + 2 * g + st, kHandOver);
            row_stage_any<GT>(2, a, 4 * tile * a.tile_q, blocks_of(tile), warp - kRowCompute / 32, kRowStagers / 32, 0, a.rows, lane,
                              tile0 + 2 * st * a.tile_q);
            fill_table(tile, tile0 + 2 * st * a.tile_q, tid - kRowCompute, kRowStagers);
            __threadfence_block();
            for (int g = 0; g < kGroups; ++g) bar_arrive(kFull + 2 * g + st, kHandOver);
        }
        __syncthreads();
        __syncthreads();
        return;
    }

    const bool active = ql < a.tq && tid < kRowCompute;      // (all warps are here where they stage together)
    float outer[kRowJT];
#pragma unroll
    for (int v = 0; v < kRowJT; ++v) {
        outer[v] = 0.f;
        if (TURN && tid < kRowCompute) totals[v * kRowCompute + tid] = 0.f;
    }
    if constexpr (TURN) {
        // Few and short variables are carried around the loop: the registers are what limits the warps of an SM.
        const int my_tiles = (int)(tile_end - tile_begin);
        const int group2 = warp / (kRowCompute / 32 / kGroups) * 2;
        const int last_blocks = my_tiles > 0 ? blocks_of(tile_end - 1) : 0;
        // the block, counted from this CTA's first, at which the high counter word changes (once in 2^32 blocks)
        const uint64_t to_change = 0x100000000ull - (first_q() & 0xFFFFFFFFull);
        int change = to_change < (uint64_t)INT_MAX ? (int)to_change : INT_MAX;
        make_jp((uint32_t)(first_q() >> 32));
        for (int i = 0; i < my_tiles; ++i) {
            const int st = i & 1;
            const int blocks = i == my_tiles - 1 ? last_blocks : a.tile_q;
            if (i >= 1) bar_sync(kFull + group2 + st, kHandOver);
            const float4 *const cur = tile0 + 2 * st * a.tile_q;
            if (active) {
                const float4 *entry = cur + 2 * ql;
                for (int upto = 0; upto < blocks;) {
                    if (upto == change - i * a.tile_q) {
                        change = INT_MAX;
                        make_jp((uint32_t)(first_q() >> 32) + 1);
                    }
                    upto = min(min(upto + kRowSumSteps * a.tq, blocks), change - i * a.tile_q);
                    float acc[kRowJT] = {};
                    for (const float4 *const stop = cur + 2 * upto; entry < stop; entry += 2 * a.tq) {
                        const float4 g = entry[0], e = entry[1];
                        QPart qp;
                        qp.hi_b = __float_as_uint(e.x);
                        qp.lo_b = __float_as_uint(e.y);
                        qp.w3 = __float_as_uint(e.z);
                        const float2 gc = make_float2(g.x, g.y), gs = make_float2(g.z, g.w);
                        uint4 w[kRowJT];
                        float2 l[kRowJT];
#pragma unroll
                        for (int v = 0; v < kRowJT; ++v) w[v] = philox_combine(jp[v], qp, a.keys);
                        bm_logs<kRowJT, true>(w, l);
#pragma unroll
                        for (int v = 0; v < kRowJT; ++v) {
                            const TurnParts r = turn_parts(w[v], l[v], turns, a.keys);
                            const float2 t = __ffma2_rn(r.n, gs, __fmul2_rn(r.c, gc));
                            acc[v] = fmaf(r.s.x, t.x, fmaf(r.s.y, t.y, acc[v]));
                        }
                    }
#pragma unroll
                    for (int v = 0; v < kRowJT; ++v) totals[v * kRowCompute + tid] += acc[v];
                }
            }
            if (i + 2 < my_tiles) bar_arrive(kEmpty + group2 + st, kHandOver);
        }
    } else {
        // The loop above, with the vectors' half formed before the first tile, cost bf16 rows staged by all warps up to 6 %: registers were
        // spilled (us, one row, d = 1.4e6: m = 2: 14.5 -> 15.5; shifted, m = 4: 17.3 -> 18.0; this loop: 14.5, 17.1).
        uint32_t jp_q_hi = 0;
        bool have_jp = false;
        for (int64_t tile = tile_begin; tile < tile_end; ++tile) {
            const int i = (int)(tile - tile_begin), st = TOGETHER ? 0 : i & 1;
            if (i >= 1) {
                if constexpr (TOGETHER) {
                    __syncthreads();                         // everyone is done with the tile
                    row_stage_any<GT>(2, a, 4 * tile * a.tile_q, blocks_of(tile), warp, kRowWarps, 0, a.rows, lane, tile0);
                    fill_table(tile, tile0, tid, kRowThreads);
                    __syncthreads();
                } else {
                    bar_sync(kFull + st, kHandOver);
                }
            }
            const float4 *cur = tile0 + 2 * st * a.tile_q;
            const int blocks = blocks_of(tile);
            const uint64_t q0 = a.q_base + (uint64_t)tile * a.tile_q;
            // the block of this tile at which the high counter word changes (once in 2^32 blocks)
            const uint64_t to_change = 0x100000000ull - (q0 & 0xFFFFFFFFull);
            int change = to_change < (uint64_t)blocks ? (int)to_change : INT_MAX;
            uint32_t q_hi = (uint32_t)(q0 >> 32);
            int qq = ql;
            if (active) {
                for (int upto = 0; upto < blocks;) {
                    if (upto == change) {
                        ++q_hi;
                        change = INT_MAX;
                    }
                    if (!have_jp || q_hi != jp_q_hi) {
                        make_jp(q_hi);
                        jp_q_hi = q_hi;
                        have_jp = true;
                    }
                    upto = min(min(upto + kRowSumSteps * a.tq, blocks), change);
                    float2 acc[kRowJT];
#pragma unroll
                    for (int v = 0; v < kRowJT; ++v) acc[v] = make_float2(0.f, 0.f);
                    const float4 *entry = cur + 2 * qq;
                    for (; qq < upto; qq += a.tq, entry += 2 * a.tq) {
                        const float4 g = entry[0], e = entry[1];
                        QPart qp;
                        qp.hi_b = __float_as_uint(e.x);
                        qp.lo_b = __float_as_uint(e.y);
                        qp.w3 = __float_as_uint(e.z);
                        uint4 w[kRowJT];
#pragma unroll
                        for (int v = 0; v < kRowJT; ++v) w[v] = philox_combine(jp[v], qp, a.keys);
                        BmParts r[kRowJT];
                        box_muller_parts<kRowJT>(w, r);
                        const float2 gc = make_float2(g.x, g.y), gs = make_float2(g.z, g.w);
#pragma unroll
                        for (int v = 0; v < kRowJT; ++v) {
                            const float2 c = __fmul2_rn(__fmul2_rn(r[v].y, r[v].sp), gc);
                            acc[v] = __ffma2_rn(r[v].s, __ffma2_rn(r[v].cs, gs, c), acc[v]);
                        }
                    }
#pragma unroll
                    for (int v = 0; v < kRowJT; ++v) outer[v] += acc[v].x + acc[v].y;
                }
            }
            if (!TOGETHER && tile + 2 < tile_end) bar_arrive(kEmpty + st, kHandOver);
        }
    }

    // The next kernel is let in only now: its CTAs, waiting beside this kernel's, would be in the way of the generating warps
    // (least-squares step at d = 8192: 102 -> 99 us).
    grid_trigger();

    // fixed-order sum over the ql lanes
    __syncthreads();
    float *red = reinterpret_cast<float *>(tile0);
    const int plane = kRowJT * a.tj;
    if (active)
#pragma unroll
        for (int v = 0; v < kRowJT; ++v) red[ql * plane + v * a.tj + jl] = TURN ? totals[v * kRowCompute + tid] : outer[v];
    __syncthreads();
    int lanes = a.tq;
    if constexpr (TURN) {
        // in two levels where there are threads for it (one would add 384 lanes at m = 8: 5 us)
        const int ranges = min(kRowCompute / plane, a.tq / 4);
        if (ranges > 1) {
            const int idx = tid % plane, range = tid / plane;
            float s = 0.f;
            if (range < ranges)
                for (int l = a.tq * range / ranges; l < a.tq * (range + 1) / ranges; ++l) s += red[l * plane + idx];
            bar_sync(kLast, kRowCompute);                    // the staging warps have gone
            if (range < ranges) red[range * plane + idx] = s;
            bar_sync(kLast, kRowCompute);
            lanes = ranges;
        }
    }
    for (int idx = tid; idx < plane; idx += kRowCompute) {
        float s = 0.f;
        for (int l = 0; l < lanes; ++l) s += red[l * plane + idx];
        if (jbase + idx < a.m) a.partial[(int64_t)blockIdx.x * a.m + jbase + idx] = TURN ? kTurnScale * s : s;
    }
}

}  // namespace

// Rows r and r + period have the same alignment; do all of them start on a 16-byte boundary?  (Of a single row that is asked too: the way
// it is staged changes no bit of the sums, and a row of odd length is staged faster the way shifted rows are, whose ends are read
// element by element from fewer lanes: d = 1567, m = 1496: 8.3 us, as an aligned row 8.9, bf16 8.8 and 9.6.)
static int row_period(int dtype, int64_t ldg) {
    int period = 1;
    while ((int64_t)period * ldg % (dtype == 1 ? 8 : 4) != 0) period *= 2;
    return period;
}
// Staging a row of a block costs more where rows have to be shifted into place; where rows are many against the
// vectors the staging warps cannot keep up and all warps stage (us, two warps -> all: n = 8, m = 8: 451 -> 375;
// n = 50, m = 21: 961 -> 728; unaligned n = 5, m = 8: 798 -> 484; but n = 32, m = 100: 1709 -> 1770).
static bool row_together(int32_t rows, bool aligned, int32_t m) { return (int64_t)rows * (aligned ? 3 : 7) >= m; }

// The table of angles pays from the microsecond it takes on, where the staging warps keep up with the faster
// generation (one in seven instead of one in five): lines through measured shapes (us, without -> with; aligned rows, d = 1e7: n = 5,
// m = 32: 537 -> 522 the round; n = 32, m = 100: 1649 -> 1584; but n = 4, m = 16: 300 -> 330, n = 8, m = 32: 539 -> 549;
// shifted, d = 1e7: n = 7, m = 64: 1073 -> 1063; n = 5, m = 100 at d = 1e6: 178 -> 171; but n = 3, m = 32: 579 -> 603,
// n = 16, m = 128: 2147 -> 2190).  By size (n = 1): d = 3e5, m = 64: 23.3 -> 21.8; d = 5e4, m = 400: 23.0 -> 22.8.  Few blocks for
// many vectors share out badly over one CTA per SM, so more than 512 vectors need three times the work: at 2^24 Gaussians m = 768: 20.0 -> 22.3,
// 4096: 20.1 -> 22.7, 8192: 20.4 -> 22.3; at 2.7 times as many -0.4, -2.4, -1.3 %.
// The message of a single row must not depend on where the row starts, so there the line asks for the number of vectors alone, and lies
// where aligned and shifted rows both gain (d = 1e7, aligned / shifted: m = 24: 216 -> 198 / 226 -> 205; but m = 13, d = 1e8: 1387 -> 1302 /
// 1548 -> 1707; m = 20, d = 3e6: 60 -> 60 / 62 -> 66).
static bool row_turn(int32_t rows, bool aligned, int32_t m, int64_t d) {
    if (d < ((int64_t)(m > 512 ? 3 : 1) << 24) / m) return false;
    if (rows == 1) return m > 20;
    return aligned ? 11 * (int64_t)rows + 40 < 4 * (int64_t)m : 8 * (int64_t)rows + 10 < m;
}

// Bytes of dynamic shared memory: two tiles with their tables (or, while the first one is staged, one and the row ranges it is
// added up from, at most a segment of 64 blocks per warp), in whose place the last sums meet; with the table of angles, it and the sums
// over tiles.
template <bool TURN>
static constexpr size_t row_shared(int tile_q, int threads) {
    const size_t tile = (size_t)tile_q * (16 + 16), ranges = (size_t)RowCta<TURN>::kWarps * 64 * 16, red = (size_t)threads * kRowJT * 4;
    const size_t stage = tile + (tile > ranges ? tile : ranges);
    return (stage > red ? stage : red) + (TURN ? kTurnBytes + kRowJT * 4 * RowCta<true>::kCompute : 0);
}
constexpr size_t kSharedPerCta = 227 * 1024, kSharedPerSm = 228 * 1024;
static_assert(row_shared<true>(RowCta<true>::kTileBlocks, RowCta<true>::kCompute) <= kSharedPerCta, "the longest tile fits a CTA");
static_assert(RowCta<false>::kPerSm * (row_shared<false>(RowCta<false>::kTileBlocks, RowCta<false>::kCompute) + 1024) <= kSharedPerSm, "and an SM");

// More than half a byte to stage per multiply of a Gaussian.
static bool row_heavy(int dtype, int32_t rows, int32_t m) { return 2 * (int64_t)rows * (dtype == 1 ? 2 : 4) > m; }

static RowPlan plan_rows(bool turn, bool heavy, int32_t m, int64_t d, int sm_count) {
    RowPlan p{};
    p.turn = turn;
    const int compute = turn ? RowCta<true>::kCompute : RowCta<false>::kCompute;
    p.compute = compute;
    const int per_sm = turn ? RowCta<true>::kPerSm : RowCta<false>::kPerSm;
    const int room = turn ? RowCta<true>::kTileBlocks : RowCta<false>::kTileBlocks;
    // Threads across vectors: one per quadruple, in as few CTA rows as keep at least 15/16 of the generating
    // threads busy (every CTA row stages the gradients again)
    const int quads = (m + kRowJT - 1) / kRowJT;
    double best = -1.0;
    for (int g = (quads + compute - 1) / compute, tried = 0; tried < 8 && g <= quads; ++g, ++tried) {
        const int tj = (quads + g - 1) / g, tq = compute / tj;
        const double busy = (double)quads / g * tq / compute;
        if (busy > best + 0.02) {
            best = busy;
            p.grid_y = g;
            p.tj = tj;
            p.tq = tq;
        }
        if (busy >= 15.0 / 16.0) break;
    }
    const int64_t nq = (d + 3) >> 2;
    int64_t slots = (int64_t)sm_count * per_sm / p.grid_y;             // CTAs across coordinates that are resident together
    if (slots < 1) slots = 1;
    // blocks per tile: as many steps per tile and generating thread as fit (1024 blocks without the table, 2048 with it: two tiles
    // take 64 or 128 KB), at most 64 or 128, and of the tile counts per CTA from there on the one that leaves the fewest steps to the
    // CTA with most of them (d = 1e6, m = 100: 104 -> 98 us).  At every tile a group's warps wait for its slowest: us, at most 32
    // steps -> this: d = 2.56e7, m = 256: one row 5006 -> 4944, eight rows 5035 -> 4987; 32 rows of 1e7, m = 1000: 7830 -> 7746; 16 bf16 rows of
    // 3.1e7, m = 1024: 24198 -> 23915; without the table, seven shifted rows of 1e7, m = 64: 595 -> 589; more steps gained nothing more.
    // Many rows with the table (row_heavy): 32, since nothing is generated before a CTA's first tile is there.  us, 32 -> 128 steps:
    // 64 rows of 4e6, m = 200: 1260 -> 1273; but 40 of 5e6, m = 357: 2770 -> 2762;
    // 64 of 2e6, m = 1000: 3025 -> 3001; 24 bf16 rows of 1e7, m = 100: 1543 -> 1534.  Not without the table, where all warps stage: 64 shifted rows
    // of 4e6, m = 200, with 32 steps instead of 64: 1409 -> 1522.
    const int steps_most = turn ? heavy ? 32 : RowCta<true>::kTileSteps : RowCta<false>::kTileSteps;
    const int64_t most = steps_most * p.tq < room ? steps_most * p.tq : room / p.tq * p.tq;
    const int64_t least_tiles = (nq + slots * most - 1) / (slots * most);
    int64_t best_steps = -1;
    for (int64_t k = least_tiles; k <= 2 * least_tiles && k < least_tiles + 16; ++k) {
        const int64_t steps = ((nq + slots * k - 1) / (slots * k) + p.tq - 1) / p.tq;
        if (best_steps < 0 || k * steps < best_steps) {
            best_steps = k * steps;
            p.tile_q = (int)(steps * p.tq);
        }
    }
    p.tiles = (nq + p.tile_q - 1) / p.tile_q;
    p.grid_x = (int)(slots < p.tiles ? slots : p.tiles);
    p.chain = chain_pays((int64_t)p.grid_x * p.grid_y, (int64_t)sm_count * per_sm, d, m);
    p.smem = turn ? row_shared<true>(p.tile_q, p.tj * p.tq) : row_shared<false>(p.tile_q, p.tj * p.tq);
    return p;
}

RowPlan make_row_plan(const void *G, int dtype, int32_t rows, int64_t ldg, int32_t m, int64_t d, int sm_count) {
    const bool aligned = row_period(dtype, ldg) == 1 && reinterpret_cast<uintptr_t>(G) % 16 == 0;
    return plan_rows(row_turn(rows, aligned, m, d), row_heavy(dtype, rows, m), m, d, sm_count);
}

int row_plan_columns(int32_t m, int64_t d, int sm_count) {
    const int with = plan_rows(true, false, m, d, sm_count).grid_x, heavy = plan_rows(true, true, m, d, sm_count).grid_x;
    const int without = plan_rows(false, false, m, d, sm_count).grid_x;
    return std::max({with, heavy, without});
}

cudaError_t launch_project_row(const RowPlan &plan, const RoundKeys &keys, uint32_t t, const void *G, int dtype, int32_t rows,
                               int64_t ldg, float scale, int64_t d, int32_t m, uint64_t q_base, float *partial,
                               cudaStream_t stream) {
    RowArgs a{};
    a.G = G;
    a.ldg = ldg;
    a.d = d;
    a.tiles = plan.tiles;
    a.q_base = q_base;
    a.partial = partial;
    a.rows = rows;
    a.period = row_period(dtype, ldg);
    a.aligned = a.period == 1 && reinterpret_cast<uintptr_t>(G) % 16 == 0 && 4 * plan.tile_q % (dtype == 1 ? 8 : 4) == 0;
    a.scale = scale;
    a.m = m;
    a.tile_q = plan.tile_q;
    a.tj = plan.tj;
    a.tq = plan.tq;
    a.t = t;
    a.keys = keys;
    const dim3 grid(plan.grid_x, plan.grid_y);
    auto go = [&](auto kernel) { return launch_chained(plan.chain, kernel, grid, dim3(plan.turn ? RowCta<true>::kThreads : RowCta<false>::kThreads), plan.smem, stream, a); };
    const bool together = row_together(rows, a.aligned, m);
    auto pick = [&](auto element) {
        using GT = decltype(element);
        if (plan.turn) return go(project_row_kernel<GT, kRowTurn>);
        return together ? go(project_row_kernel<GT, kRowTogether>) : go(project_row_kernel<GT, kRowShort>);
    };
    return dtype == 1 ? pick(__nv_bfloat16{}) : pick(float{});
}

}  // namespace core
