// Fused regenerate-and-reconstruct kernel: gtilde[k] = (1/m) sum_j pbar[j] xi_j[k]
// (Algorithm 1, receiver's step; the equation that follows Algorithm 1).
//
// A thread owns one or two blocks of four coordinates and runs over the vectors j,
// regenerating xi_j for them from the same counters the projection used.  The
// part of the Philox evaluation that depends only on the block is computed once per
// thread; the part that depends only on j is tabulated per CTA in shared memory next
// to pbar[j], so the loop reads one 16-byte broadcast per j.  Every output coordinate
// is written exactly once, as a 16-byte store where alignment allows.
#include "core_emit.cuh"
#include "core_finish.cuh"
#include "core_internal.h"
#include "core_sync.cuh"

namespace core {

namespace {

constexpr int kWideUQ = 2;                        // the kernel for few or very many vectors: coordinate blocks per thread,
constexpr int kWideQ = kThreads * kWideUQ;        // per CTA step,
constexpr int kWideJStep = 2;                     // vectors generated together,
constexpr int kWideCtas = 3;                      // resident CTAs per SM (register-limited)
constexpr int kJChunk = 2048;                     // vectors tabulated at a time (32 KB)
constexpr int kTurnWarps = 32;                    // the kernel for long vectors: one CTA per SM
constexpr int kTurnJStep = 4;                     // vectors generated together
constexpr int kTurnVectors = 8192;                // most vectors it takes: their table has 128 KB
constexpr int kTurnShares = kTurnWarps * 32 * 16;

struct ReconstructArgs {
    float *pbar;
    MessageParts parts;        // partial != nullptr: the message is formed here (short vectors only)
    float *out;
    int64_t k_begin;
    int64_t k_end;
    int m;
    int vec_ok;       // out (and the epilogue arrays) + 4*(q - q_begin) are 16-byte aligned
    uint32_t t;
    RoundKeys keys;
    ReconstructEpilogue epi;   // base == nullptr: store the estimate itself
};

// acc[u] += sum over JS consecutive table entries of pbar[j] * xi_j[block u], j ascending.
template <int JS, int UQ>
__device__ __forceinline__ void rec_step(const uint4 *entries, const QPart (&qp)[UQ], const RoundKeys &keys, float4 (&acc)[UQ]) {
    uint4 w[JS * UQ];
    float p[JS];
#pragma unroll
    for (int s = 0; s < JS; ++s) {
        const uint4 e = entries[s];
        p[s] = __uint_as_float(e.w);
        JPart jp;
        jp.x0 = e.x;
        jp.x2 = e.y;
        jp.w3 = e.z;
#pragma unroll
        for (int u = 0; u < UQ; ++u) w[s * UQ + u] = philox_combine(jp, qp[u], keys);
    }
    BmParts r[JS * UQ];
    box_muller_parts<JS * UQ>(w, r);
    // pbar_j xi_j with the message meeting the radius first: ((pbar S) y) sp and (pbar S) cs, four packed
    // instructions per call instead of five, and xi_j itself (pbar = 1) bit for bit what the projection
    // multiplies with.  Accumulator lanes: (x, z) = cosine lanes of pair a, b; (y, w) = sine lanes.
#pragma unroll
    for (int s = 0; s < JS; ++s) {
#pragma unroll
        for (int u = 0; u < UQ; ++u) {
            const BmParts rr = r[s * UQ + u];
            const float2 ps = __fmul2_rn(make_float2(p[s], p[s]), rr.s);
            const float2 psy = __fmul2_rn(ps, rr.y);
            const float2 c2 = __ffma2_rn(psy, rr.sp, make_float2(acc[u].x, acc[u].z));
            const float2 s2 = __ffma2_rn(ps, rr.cs, make_float2(acc[u].y, acc[u].w));
            acc[u] = make_float4(c2.x, s2.x, c2.y, s2.y);
        }
    }
}

// The same for one block, with the angles from the table (values short of the factor kTurnScale, which sits in the message):
// three packed instructions per call.  Lanes of the accumulators = pair a, pair b.  The products of a step are added up before
// they meet the accumulator: rounding errors grow with the square root of a chain's length (m = 500: relative error 2.9e-7
// in one chain of all vectors).
template <int JS>
__device__ __forceinline__ void turn_step(const uint4 *entries, const float2 *turns, const QPart &qp, const RoundKeys &keys,
                                          float2 &cosine, float2 &sine) {
    uint4 w[JS];
    float2 l[JS];
    float p[JS];
#pragma unroll
    for (int s = 0; s < JS; ++s) {
        const uint4 e = entries[s];
        p[s] = __uint_as_float(e.w);
        JPart jp;
        jp.x0 = e.x;
        jp.x2 = e.y;
        jp.w3 = e.z;
        w[s] = philox_combine(jp, qp, keys);
    }
    bm_logs<JS, true>(w, l);
    float2 c, n;
#pragma unroll
    for (int s = 0; s < JS; ++s) {
        const TurnParts r = turn_parts(w[s], l[s], turns, keys);
        const float2 ps = __fmul2_rn(make_float2(p[s], p[s]), r.s);
        c = s == 0 ? __fmul2_rn(ps, r.c) : __ffma2_rn(ps, r.c, c);
        n = s == 0 ? __fmul2_rn(ps, r.n) : __ffma2_rn(ps, r.n, n);
    }
    cosine = __fadd2_rn(cosine, c);
    sine = __fadd2_rn(sine, n);
}

// Long vectors.  One CTA per SM takes an equal share of the vector in units of 32 blocks, one per lane.  Its warps
// run through whole units by themselves; the last one to two units per warp are cut evenly over the warps as one long line of
// (unit, vector) pairs, so that no warp waits for others at the end: a unit that several warps share is added up, in the
// order of its vectors, by the one that has its first.  The table of angles is made while the previous kernel ends.
// us, this kernel against 512 blocks per CTA and step with the polynomials (d < 2.4e6: against the kernel below): d = 2.5e7,
// m = 256: 5205 -> 4728; d = 1e8, m = 64: 5111 -> 4687; d = 1e6, m = 100: 86.9 -> 77.3.  (24 warps: 0.2 to 1 % slower; two blocks
// per lane and two vectors per step in place of one and four: equal in long vectors, 2 to 5 % slower at d = 1e6; passes over
// the CTA's share by all of its threads instead of the line: up to 15 % slower at d = 1e6; partial sums of 64 vectors in
// shared memory instead of sums over a step: 1.4 % slower.)
struct TurnPlan {                                  // of the units that share the high counter word: all of a CTA's, but once in 2^32 blocks
    uint32_t q_lo, q_hi;                           // first block
    int units;
    int rounds;                                    // whole units per warp before the line
    int2 start[kTurnWarps + 1];                    // {unit, vector} where warp w's share of the line starts
};

__global__ void __launch_bounds__(kTurnWarps * 32, 1)
reconstruct_kernel(const __grid_constant__ ReconstructArgs a) {
    grid_trigger();
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *const turns = reinterpret_cast<float2 *>(smem);
    float4 *const shares = reinterpret_cast<float4 *>(smem + kTurnBytes);  // [thread]: a warp's share of its first unit
    uint4 *const table = reinterpret_cast<uint4 *>(shares + kTurnWarps * 32);     // {JPart.x0, JPart.x2, JPart.w3, kTurnScale pbar[j]}
    // What is not needed while Gaussians are made stays in shared memory: the generating loop wants all 64 registers.
    __shared__ TurnPlan plan_memory;
    volatile TurnPlan &plan = plan_memory;
    fill_turn_table<kTurnWarps>(turns, threadIdx.x >> 5, threadIdx.x & 31);
    grid_wait();
    auto emit = [&](int unit, float4 s) {
        const uint64_t q_begin = (uint64_t)a.k_begin >> 2, q_end = ((uint64_t)a.k_end + 3) >> 2;
        const uint64_t q = ((uint64_t)plan.q_hi << 32) + plan.q_lo + (uint32_t)(unit * 32) + (threadIdx.x & 31);
        const float inv_m = 1.0f / (float)a.m;
        if (q < q_end) emit_block(a, q, q_begin, make_float4(s.x * inv_m, s.y * inv_m, s.z * inv_m, s.w * inv_m));
    };
    const int64_t all = (int64_t)((((uint64_t)a.k_end + 3) >> 2) - ((uint64_t)a.k_begin >> 2) + 31) >> 5;
    for (int64_t unit0 = all * blockIdx.x / gridDim.x; unit0 < all * (blockIdx.x + 1) / gridDim.x; unit0 += plan.units) {
        __syncthreads();                                                   // everyone is done with the previous plan and table
        const uint64_t q0 = ((uint64_t)a.k_begin >> 2) + ((uint64_t)unit0 << 5);
        const int units = (int)min(all * (blockIdx.x + 1) / gridDim.x - unit0, (int64_t)((0x100000000ull - (q0 & 0xFFFFFFFFull)) >> 5));
        const int rounds = max(units / kTurnWarps - 1, 0);
        if (threadIdx.x <= kTurnWarps) {
            const int64_t at = (int64_t)threadIdx.x * (units - rounds * kTurnWarps) * a.m / kTurnWarps;
            const int unit = (int)(at / a.m);
            plan.start[threadIdx.x].x = unit + rounds * kTurnWarps;
            plan.start[threadIdx.x].y = (int)(at - (int64_t)unit * a.m) / kTurnJStep * kTurnJStep;
            if (threadIdx.x == 0) {
                plan.q_lo = (uint32_t)q0;
                plan.q_hi = (uint32_t)(q0 >> 32);
                plan.units = units;
                plan.rounds = rounds;
            }
        }
        for (int j = threadIdx.x; j < a.m; j += kTurnWarps * 32) {
            const JPart jp = philox_jpart((uint32_t)j, (uint32_t)(q0 >> 32), a.keys);
            table[j] = make_uint4(jp.x0, jp.x2, jp.w3, __float_as_uint(kTurnScale * __ldcg(a.pbar + j)));
        }
        __syncthreads();
        bool head = false;                                                 // has the first vectors of a unit, others the rest
        float4 s;
        for (int r = 0;; ++r) {
            // whole unit r of this warp, or segment r - rounds of its share of the line
            const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
            auto segment = [&](int &unit, int &j_begin, int &j_end) {
                const int line = r - plan.rounds;
                unit = r * kTurnWarps + warp;
                j_begin = 0;
                j_end = a.m;
                if (line < 0) return true;
                unit = plan.start[warp].x + line;
                if (line == 0) j_begin = plan.start[warp].y;
                const int end = plan.start[warp + 1].x;
                if (unit == end) j_end = plan.start[warp + 1].y;
                return unit < end || (unit == end && j_begin < j_end);
            };
            int unit, j_begin, j_end;
            if (!segment(unit, j_begin, j_end)) break;
            const QPart qp = philox_qpart(plan.q_lo + (uint32_t)(unit * 32) + (threadIdx.x & 31), a.t, a.keys);
            float2 cosine = make_float2(0.f, 0.f), sine = make_float2(0.f, 0.f);
            const uint4 *entry = table + j_begin, *const stop = table + j_end;
            for (; entry + kTurnJStep <= stop; entry += kTurnJStep) turn_step<kTurnJStep>(entry, turns, qp, a.keys, cosine, sine);
            for (; entry < stop; ++entry) turn_step<1>(entry, turns, qp, a.keys, cosine, sine);
            s = make_float4(cosine.x, sine.x, cosine.y, sine.y);
            segment(unit, j_begin, j_end);                                 // again: not kept in registers meanwhile
            if (j_begin > 0) {
                shares[threadIdx.x] = s;
            } else if (j_end == a.m) {
                emit(unit, s);
            } else {
                head = true;
                break;
            }
        }
        __syncthreads();
        if (head) {
            const int warp = threadIdx.x >> 5, unit = plan.start[warp + 1].x;
            for (int v = warp + 1; v < kTurnWarps && plan.start[v].x == unit; ++v) {     // the warps that start inside this unit
                if (plan.start[v + 1].x == unit && plan.start[v + 1].y == plan.start[v].y) continue;        // with nothing of it
                const float4 p = shares[v * 32 + (threadIdx.x & 31)];
                s = make_float4(s.x + p.x, s.y + p.y, s.z + p.z, s.w + p.w);
            }
            emit(unit, s);
        }
    }
}

// Long vectors where the table of angles does not pay: few vectors, whose Gaussians cost less than the stores and the table, or more
// vectors than fit beside it.  512 blocks per CTA and step, two per thread, three CTAs per SM that walk over the vector; where the
// vectors are more than kJChunk their table is made anew for every chunk.
__global__ void __launch_bounds__(kThreads, kWideCtas)
reconstruct_wide_kernel(const __grid_constant__ ReconstructArgs a) {
    grid_trigger();
    grid_wait();
    __shared__ uint4 table[kJChunk];              // {JPart.x0, JPart.x2, JPart.w3, bits of pbar[j]}
    const int tid = threadIdx.x;
    const uint64_t q_begin = (uint64_t)a.k_begin >> 2;
    const uint64_t q_end = ((uint64_t)a.k_end + 3) >> 2;
    const uint64_t groups = (q_end - q_begin + kWideQ - 1) / kWideQ;
    const float inv_m = 1.0f / (float)a.m;

    bool have_table = false;
    uint32_t table_qhi = 0;

    for (uint64_t grp = blockIdx.x; grp < groups; grp += gridDim.x) {
        // q_begin is a multiple of kWideQ (launch_reconstruct checks), so a group never
        // straddles a multiple of 2^32 and all its blocks share the high counter word.
        const uint64_t gq0 = q_begin + grp * kWideQ;
        const uint32_t grp_qhi = (uint32_t)(gq0 >> 32);

        float4 acc[kWideUQ];
        QPart qp[kWideUQ];
        uint64_t qv[kWideUQ];
#pragma unroll
        for (int u = 0; u < kWideUQ; ++u) {
            qv[u] = gq0 + (uint64_t)(tid + u * kThreads);
            qp[u] = philox_qpart((uint32_t)qv[u], a.t, a.keys);
            acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        }

        for (int j0 = 0; j0 < a.m; j0 += kJChunk) {
            const int jn = min(kJChunk, a.m - j0);
            if (!have_table || table_qhi != grp_qhi || a.m > kJChunk) {
                __syncthreads();                  // everyone is done with the previous table
                for (int jj = tid; jj < jn; jj += kThreads) {
                    const JPart jp = philox_jpart((uint32_t)(j0 + jj), grp_qhi, a.keys);
                    table[jj] = make_uint4(jp.x0, jp.x2, jp.w3, __float_as_uint(__ldcg(a.pbar + j0 + jj)));
                }
                __syncthreads();
                have_table = true;
                table_qhi = grp_qhi;
            }
            int jj = 0;
            for (; jj + kWideJStep <= jn; jj += kWideJStep) rec_step<kWideJStep, kWideUQ>(table + jj, qp, a.keys, acc);
            for (; jj < jn; ++jj) rec_step<1, kWideUQ>(table + jj, qp, a.keys, acc);
        }

#pragma unroll
        for (int u = 0; u < kWideUQ; ++u) {
            if (qv[u] >= q_end) continue;
            emit_block(a, qv[u], q_begin, make_float4(acc[u].x * inv_m, acc[u].y * inv_m, acc[u].z * inv_m, acc[u].w * inv_m));
        }
    }
}

// Short vectors: the kernels above would leave most of their warps without work (d = 8192 is 64 units),
// so here the SLICES warp groups of a CTA share out the vectors of 256 / SLICES blocks; the partial sums
// of a block meet in shared memory and are added in ascending order of the vector ranges.  Few vectors
// get few slices (a slice wants at least four vectors to generate together); where even eight slices leave SMs
// idle and vectors are many, a cluster of up to eight CTAs shares them out as well, and the first one adds up.
constexpr int kJoinVectors = 512;                  // most vectors whose message is formed here: the rest of the
constexpr int kJoinEntries = (kJChunk - kJoinVectors) * 16 / 4 / kFinishSlices;     // table takes the slices of n * m entries

__device__ __forceinline__ void store_cluster(const void *smem, uint32_t rank, float4 v) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(smem)), "r"(rank));
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(remote), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

template <int SLICES>
__global__ void __launch_bounds__(kThreads, 4)
reconstruct_small_kernel(const __grid_constant__ ReconstructArgs a) {
    grid_trigger();
    constexpr int QB = kThreads / SLICES;          // blocks per CTA
    constexpr int RANKS = SLICES == 8 ? 8 : 1;     // CTAs of a cluster at most
    __shared__ uint4 table[kJChunk];               // as above
    __shared__ float4 part[SLICES][QB];
    __shared__ float4 inbox[RANKS][QB];
    const int tid = threadIdx.x, ql = tid % QB, slice = tid / QB;
    uint32_t rank = 0, ranks = 1;
    if constexpr (RANKS > 1) {
        rank = cluster_rank();
        asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(ranks));
        cluster_arrive();                          // this CTA has started
    }
    const uint64_t q_begin = (uint64_t)a.k_begin >> 2;
    const uint64_t q_end = ((uint64_t)a.k_end + 3) >> 2;
    const uint64_t q0 = q_begin + (uint64_t)(blockIdx.x / ranks) * QB;     // multiple of 32: one high counter word per CTA
    const uint32_t q_hi = (uint32_t)(q0 >> 32);
    const uint64_t q = q0 + (uint64_t)ql;
    const QPart qp[1] = {philox_qpart((uint32_t)q, a.t, a.keys)};
    float4 acc[1] = {make_float4(0.f, 0.f, 0.f, 0.f)};
    const int mine = ((a.m + (int)ranks - 1) / (int)ranks + 3) & ~3;       // vectors of this CTA
    const int m_begin = min((int)rank * mine, a.m), m_end = min(m_begin + mine, a.m);
    for (int j0 = m_begin; j0 < m_end; j0 += kJChunk) {
        const int jn = min(kJChunk, m_end - j0);
        if (j0 > m_begin) __syncthreads();         // everyone is done with the previous table
        for (int jj = tid; jj < jn; jj += kThreads) {
            const JPart jp = philox_jpart((uint32_t)(j0 + jj), q_hi, a.keys);
            table[jj] = make_uint4(jp.x0, jp.x2, jp.w3, 0u);
        }
        if (j0 == m_begin) grid_wait();            // the message comes last
        if (a.parts.partial) {
            const int n = a.parts.n, entries = n * jn;
            float *const slices = reinterpret_cast<float *>(table + kJoinVectors);
            for (int e = tid; e < entries * kFinishSlices; e += kThreads) {
                const int entry = e % entries, i = entry / jn, j = entry % jn;
                // (eight in flight while there are; sixteen, or eight for the last ones too, would spill)
                slices[e] = finish_slice<4, 8>(a.parts.partial, a.parts.chunks, (int64_t)n * a.m, (int64_t)i * a.m + j0 + j, e / entries);
            }
            __syncthreads();
            for (int jj = tid; jj < jn; jj += kThreads) {
                float sum = 0.f;
                for (int i = 0; i < n; ++i) sum += finish_join(slices + i * jn + jj, entries);
                sum /= (float)n;
                table[jj].w = __float_as_uint(sum);
                if (blockIdx.x < ranks) a.pbar[j0 + jj] = sum;
            }
        } else {
            for (int jj = tid; jj < jn; jj += kThreads) table[jj].w = __float_as_uint(__ldcg(a.pbar + j0 + jj));
        }
        __syncthreads();
        const int per = (jn + SLICES - 1) / SLICES;                         // vectors per slice
        const int j_begin = min(slice * per, jn), j_end = min(j_begin + per, jn);
        int jj = j_begin;
        for (; jj + 4 <= j_end; jj += 4) rec_step<4, 1>(table + jj, qp, a.keys, acc);
        for (; jj < j_end; ++jj) rec_step<1, 1>(table + jj, qp, a.keys, acc);
    }
    if (m_begin >= m_end) grid_wait();             // a CTA without vectors
    part[slice][ql] = acc[0];
    __syncthreads();
    float4 s = part[0][ql];
    if (slice == 0) {
#pragma unroll
        for (int r = 1; r < SLICES; ++r) {
            const float4 p = part[r][ql];
            s = make_float4(s.x + p.x, s.y + p.y, s.z + p.z, s.w + p.w);
        }
    }
    if constexpr (RANKS > 1) {
        cluster_wait();                            // the first CTA has started
        if (ranks > 1) {
            if (slice == 0 && rank > 0) store_cluster(&inbox[rank][ql], 0, s);
            cluster_arrive();
            cluster_wait();
            if (rank > 0) return;
            if (slice == 0)
                for (int r = 1; r < (int)ranks; ++r) {
                    const float4 p = inbox[r][ql];
                    s = make_float4(s.x + p.x, s.y + p.y, s.z + p.z, s.w + p.w);
                }
        }
    }
    if (slice == 0 && q < q_end) {
        const float inv_m = 1.0f / (float)a.m;
        emit_block(a, q, q_begin, make_float4(s.x * inv_m, s.y * inv_m, s.z * inv_m, s.w * inv_m));
    }
}

struct DebugArgs {
    uint64_t q0;
    int64_t nq;
    uint32_t j;
    uint32_t t;
    RoundKeys keys;
};

__global__ void debug_philox_kernel(const __grid_constant__ DebugArgs a, uint4 *words) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < a.nq; r += stride) {
        const uint64_t q = a.q0 + (uint64_t)r;
        words[r] = philox4x32_10((uint32_t)q, (uint32_t)(q >> 32), a.j, a.t, a.keys);
    }
}

// Goes through the split evaluation of Philox, which all round kernels use, and the polynomials of those without the table of angles.
// (The Gaussians of those with it are read back by messages and gradients that are unit vectors.)
__global__ void debug_gaussians_kernel(const __grid_constant__ DebugArgs a, float4 *z) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < a.nq; r += stride) {
        const uint64_t q = a.q0 + (uint64_t)r;
        const JPart jp = philox_jpart(a.j, (uint32_t)(q >> 32), a.keys);
        const QPart qp = philox_qpart((uint32_t)q, a.t, a.keys);
        z[r] = box_muller4(philox_combine(jp, qp, a.keys));
    }
}

__global__ void debug_box_muller_kernel(const uint4 *__restrict__ words, int64_t nb, float4 *z) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nb; r += stride)
        z[r] = box_muller4(words[r]);
}

unsigned grid_for(int64_t items, int threads, int cap) {
    int64_t g = (items + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (unsigned)g;
}

}  // namespace

// The kernel with the table of angles wants five units per SM (six in one SM and five in another are 13 % apart; at four the one for
// short vectors, with its clusters, is ahead) and work for the microsecond or two that its table takes: us, the one for short
// vectors -> this one, d = 1e5, m = 64: 9.1 -> 9.8, m = 256: 26.3 -> 25.5; d = 1e6, m = 8: 10.3 -> 11.5, m = 32: 31.0 -> 29.4; d = 3e6,
// m = 8: 25.0 -> 24.2; d = 4e4, m = 1024: 45.6 -> 47.1.  With few vectors it takes as much more work to be ahead of the wide
// kernel (m = 6, d = 3.6e6: 21.9 -> 23.1, 9.8e6: 1 % ahead), with up to three it never is (m = 1, d = 1e8: 157.8 -> 168.3; m = 2: 233 -> 244;
// m = 3, d = 2e7: 64.9 -> 67.1).  Other vectors of eight wide steps per SM or more take the wide kernel (the one for short
// vectors there: m = 1, d = 1e7: 17.4 -> 33.2; m = 4, d = 3e6: 14.7 -> 17.9).
RecKernel reconstruct_kernel_for(int64_t nq, int32_t m, int sm_count) {
    const int64_t work = (int64_t)(m < 8 ? 3 : 1) << 22;
    if (m > 3 && m <= kTurnVectors && nq >= 160 * (int64_t)sm_count && nq >= work / m) return RecKernel::kTurn;
    return (nq + kWideQ - 1) / kWideQ >= 8 * (int64_t)sm_count ? RecKernel::kWide : RecKernel::kShort;
}
// Every CTA forms the whole message: worth it while that is at most eight loads per thread (with 32, d = 8192 and m = 64, the
// launch it saves was the cheaper one: 100.7 against 105.9 us a step) and the CTAs are those of a short vector (m = 1, d = 1.6e7: 15625
// of them form it 15625 times: a round of one machine 121 -> 524).
bool reconstruct_joins(int chunks, int32_t n, int32_t m, int64_t d, int sm_count) {
    return m <= kJoinVectors && (int64_t)n * m <= kJoinEntries && (int64_t)chunks * n * m <= 2048 &&
           reconstruct_kernel_for((d + 3) >> 2, m, sm_count) == RecKernel::kShort;
}

cudaError_t launch_reconstruct(const RoundKeys &keys, uint32_t t, float *pbar, int32_t m,
                               int64_t k_begin, int64_t k_end, float *out, int sm_count,
                               cudaStream_t stream, const ReconstructEpilogue *epilogue, const MessageParts *parts) {
    if (k_end <= k_begin) return cudaSuccess;
    if (k_begin % 2048 != 0) return cudaErrorInvalidValue;
    ReconstructArgs a{};
    a.pbar = pbar;
    a.out = out;
    a.k_begin = k_begin;
    a.k_end = k_end;
    a.m = m;
    uintptr_t align = reinterpret_cast<uintptr_t>(out);
    if (epilogue && epilogue->base) {
        a.epi = *epilogue;
        align |= reinterpret_cast<uintptr_t>(epilogue->base);
        if (epilogue->shift_dst)
            align |= reinterpret_cast<uintptr_t>(epilogue->shift_src) | reinterpret_cast<uintptr_t>(epilogue->shift_dst);
    }
    a.vec_ok = (align % 16) == 0 ? 1 : 0;
    a.t = t;
    a.keys = keys;
    const int64_t nq = ((k_end + 3) >> 2) - (k_begin >> 2);
    if (parts) a.parts = *parts;
    const RecKernel kernel = reconstruct_kernel_for(nq, m, sm_count);
    if (kernel == RecKernel::kShort) {
        // more slices = fewer blocks per CTA = more CTAs: as many as it takes to go round evenly (four are resident per
        // SM), while a slice keeps at least four vectors, or sixteen where it is only for the last wave's sake
        int slices = 1, ranks = 1;
        auto ctas_with = [&](int s) { return nq / (kThreads / s); };
        while (slices < 8 && m >= 8 * slices &&
               (ctas_with(slices) < 4 * (int64_t)sm_count || (ctas_with(slices) < 16 * (int64_t)sm_count && m >= 32 * slices)))
            slices *= 2;
        const int64_t ctas = (nq + kThreads / slices - 1) / (kThreads / slices);
        if (slices == 8) {
            // CTAs of the fullest SM, each with 1 / ranks of the vectors and the work of starting up (about six vectors a
            // thread); every slice keeps eight vectors
            auto cost = [&](int r) { return (double)((ctas * r + sm_count - 1) / sm_count) * (1.0 / r + 48.0 / m); };
            for (int r = 2; r <= 8 && m >= 64 * r; ++r)
                if (cost(r) < cost(ranks)) ranks = r;
        }
        const bool chain = chain_pays(ctas * ranks, 4 * (int64_t)sm_count, 4 * nq, m);
        auto go = [&](auto kernel) {
            const ChainedLaunch launch(chain, dim3((unsigned)(ctas * ranks)), dim3(kThreads), 0, stream, ranks);
            return cudaLaunchKernelEx(&launch.cfg, kernel, a);
        };
        switch (slices) {
            case 8: return go(reconstruct_small_kernel<8>);
            case 4: return go(reconstruct_small_kernel<4>);
            case 2: return go(reconstruct_small_kernel<2>);
            default: return go(reconstruct_small_kernel<1>);
        }
    }
    if (kernel == RecKernel::kWide) {
        const int64_t steps = (nq + kWideQ - 1) / kWideQ, ctas = (int64_t)sm_count * kWideCtas;
        return launch_chained(true, reconstruct_wide_kernel, dim3((unsigned)(steps < ctas ? steps : ctas)), dim3(kThreads), 0, stream, a);
    }
    const size_t smem = kTurnBytes + kTurnShares + sizeof(uint4) * (size_t)m;
    return launch_chained(true, reconstruct_kernel, dim3((unsigned)sm_count), dim3(kTurnWarps * 32), smem, stream, a);
}

cudaError_t launch_debug_philox(const RoundKeys &keys, uint32_t t, uint32_t j, uint64_t q0, int64_t nq,
                                uint32_t *words, cudaStream_t stream) {
    if (nq <= 0) return cudaSuccess;
    DebugArgs a{q0, nq, j, t, keys};
    debug_philox_kernel<<<grid_for(nq, 256, 148 * 8), 256, 0, stream>>>(a, reinterpret_cast<uint4 *>(words));
    return cudaGetLastError();
}

cudaError_t launch_debug_gaussians(const RoundKeys &keys, uint32_t t, uint32_t j, uint64_t q0, int64_t nq,
                                   float *z, cudaStream_t stream) {
    if (nq <= 0) return cudaSuccess;
    DebugArgs a{q0, nq, j, t, keys};
    debug_gaussians_kernel<<<grid_for(nq, 256, 148 * 8), 256, 0, stream>>>(a, reinterpret_cast<float4 *>(z));
    return cudaGetLastError();
}

cudaError_t launch_debug_box_muller(const uint32_t *words, int64_t nb, float *z, cudaStream_t stream) {
    if (nb <= 0) return cudaSuccess;
    debug_box_muller_kernel<<<grid_for(nb, 256, 148 * 8), 256, 0, stream>>>(
        reinterpret_cast<const uint4 *>(words), nb, reinterpret_cast<float4 *>(z));
    return cudaGetLastError();
}

}  // namespace core
