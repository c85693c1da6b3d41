// One pass over the data matrices of the least-squares objective: for every row r of every machine
// res = A[r] . x - b[r], and either acc += res * A[r] (machine gradients, Algorithm 2's local computation) or
// loss += res^2 (the objective).  A is read from HBM once; it is the bound (4 bytes per two multiply-adds).
//
// The rows of all machines are one matrix of n * rows rows, cut evenly over one CTA per SM, whatever n and rows
// are: a CTA's range may end inside a machine and go on in the next.  Groups of W warps take the CTA's rows in
// turn: W = 1 up to 512 columns, then 2, 4, 8 and 16 up to 16384; beyond, a cluster of 2 to 8 CTAs shares the
// columns of a row.  Lane l of warp w of a group owns columns l + 32 (w + W c): x and the partial gradient of those
// columns stay in registers for the whole pass, the row's values between its dot product and its update.  Each
// group has a ring of row buffers in shared memory filled by bulk copies (one lane issues them; they start and end
// on 16-byte boundaries around the rows, so that rows of any alignment move at full rate; single columns per lane
// need no alignment either, and 16-byte reads were not faster).  Rows of up to 512 columns are handled 2 to 16 at a
// time, their dot products reduced together by a transposing butterfly (16 rows: 16 shuffles instead of 80).  In a
// cluster every warp sends its share of the dot product to all CTAs (asynchronous remote stores counted by a barrier
// there).  Every sum has a fixed order.
//
// Measured (us; pass alone unless said otherwise; before: the kernels this one replaced): n = 50, 1200 x 784: 155 -> 38;
// n = 50, 11620 x 54: gradients 377 -> 31, loss 212 -> 28; n = 16, 256 x 20000: gradients 133 -> 72; n = 8, 2048 x 8192
// (537 MB): loss 107 -> 88, gradients 87 -> 92.  Tried: cp.async instead of bulk copies (20 % slower), rings of 96 to
// 192 KB (equal), evict_normal instead of evict_first (3 to 10 us slower), 8 warps for one-warp rows (25 % slower).
#include "core_finish.cuh"
#include "core_internal.h"
#include "core_sync.cuh"

#include <algorithm>
#include <type_traits>

namespace core {

namespace {

constexpr int kPassMaxSlots = 8;
constexpr int kPassMaxWarps = 16;
constexpr int kPassOneWarp = 512;                       // columns up to which one warp holds a row
constexpr int kPassMaxCluster = 8;
constexpr int kPassCtaCols = 32 * 32 * kPassMaxWarps;   // columns a CTA can hold: 32 per lane
constexpr uint32_t kPassFlushBytes = 32u * 1024u;       // room for the groups' sums while the rings are in use
constexpr uint32_t kPassRingBytes = 128u * 1024u;       // bytes in flight per SM

// Rows at a time.  One warp per row: as many as 32 registers per lane hold.  Several: the chain from a row's arrival to
// its update crosses the CTA (about 1600 cycles), so two rows go through it together, four where up to 24 columns
// per lane leave the registers, and rows of up to 24 KB the shared memory, for it (gradients, us: 16 x 2048 rows of
// 2049 columns: 125 with one, 84 with two, 66 with four; 8 x 1500 x 5500: 56 with two, 46 with four); the 512-thread
// kernel of 16 warps per row has registers for two up to 24 columns, and gains by two up to 28, as far as the shared memory has
// room for two slots of them (14064 columns) and the rows are many enough (make_ls_pass), although some registers are then spilled (8 x 64 rows of 100000: 80 with one, 70 with two; 16 x 512
// of 14000: 89, 80).
constexpr int pass_batch(int warps_per_row, int columns) {
    return warps_per_row == 1 ? (columns <= 2 ? 16 : 32 / columns) : warps_per_row == 16 ? (columns > 28 ? 1 : 2) : columns <= 24 ? 4 : 2;
}

__device__ int g_pass_status;                           // 0, or the code of a wait that ran out

struct PassArgs {
    const float *A;
    const float *b;
    const float *x;
    const float *x_prev;     // not null: evaluate at x + gamma (x - x_prev)
    float gamma;
    int64_t d;
    int64_t rows;            // per machine; all rows of all machines when the machines are not kept apart
    int64_t total;           // n * rows
    int64_t units;           // CTAs (clusters) the rows are cut over
    float *part;             // gradients: part[slot * ldp + column]
    int64_t ldp;
    int slots_per_machine;
    double *loss_part;       // objective: one sum of squares per unit
    int cluster;             // CTAs per row
    int slice;               // columns per CTA of a cluster
    int chunk_rows;          // rows per ring slot, at most 32
    int slots;               // ring slots per group
    uint32_t slot_bytes;
    uint32_t row_stride;     // bytes between the rows of a slot; agrees with d * 4 modulo 16
    uint32_t ring_offset;    // of the rings in shared memory, behind a buffer for the groups' sums where machines are kept apart
    int flush_floats;        // room for the groups' sums: that buffer, or the rings once the last row is done
    int reverse;             // rows from the last to the first (what an ascending pass left in L2 comes first)
    int hold_back;           // test: chunks from this one on are never copied (by the first CTA of a cluster)
};

// What is read of A, as the kernel computes it and ls_pass_reads checks it on the host.
// Rows [lo, lo + count) of all machines' rows are a unit's.  `edge`: A ends less than 16 bytes before or behind them, so
// that rounding out to 16 bytes might reach beyond it (not only for the first and the last unit: rows may be one float).
struct UnitRows {
    int64_t lo;
    int count;
    bool edge;
};
__host__ __device__ inline UnitRows unit_rows(int64_t total, int64_t units, int64_t unit, int64_t d) {
    const int64_t lo = total * unit / units, hi = total * (unit + 1) / units;
    return {lo, (int)(hi - lo), lo * d < 4 || (total - hi) * d < 4};
}
// The bytes [from, to) rounded out to the 16-byte units a bulk copy moves ...
struct BulkRange {
    uintptr_t b0, b1;
};
__host__ __device__ inline BulkRange bulk_range(uintptr_t from, uintptr_t to) { return {from & ~(uintptr_t)15, (to + 15) & ~(uintptr_t)15}; }
// ... and without a first or last one that would reach beyond A (whose elements are copied one by one).
__host__ __device__ inline BulkRange bulk_range_inside(BulkRange r, uintptr_t a_begin, uintptr_t a_end) {
    return {r.b0 < a_begin ? r.b0 + 16 : r.b0, r.b1 > a_end ? r.b1 - 16 : r.b1};
}
// What a prefetch of them asks for (not at an edge).
__host__ __device__ inline BulkRange prefetch_range(uintptr_t from, uint32_t bytes) {
    return {from & ~(uintptr_t)15, (from & ~(uintptr_t)15) + (bytes & ~15u)};
}

__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}
// v to `addr` of CTA `rank` of the cluster; its 4 bytes are counted on the barrier at `bar` there.
__device__ __forceinline__ void send_remote(uint32_t addr, uint32_t bar, uint32_t rank, float v) {
    asm volatile(
        "{\n\t.reg .b32 ra, rb;\n\t"
        "mapa.shared::cluster.u32 ra, %0, %2;\n\t"
        "mapa.shared::cluster.u32 rb, %1, %2;\n\t"
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [ra], %3, [rb];\n\t}"
        ::"r"(addr), "r"(bar), "r"(rank), "r"(__float_as_uint(v))
        : "memory");
}
__device__ __forceinline__ float load_shared(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void store_shared(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }

// Sums of RB values over the warp at once: afterwards every lane holds the sum of value lane * RB / 32.
template <int RB>
__device__ __forceinline__ float butterfly(float (&p)[RB], int lane) {
    int off = 16;
#pragma unroll
    for (int half = RB / 2; half > 0; half /= 2, off /= 2) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const float send = upper ? p[k] : p[k + half];
            const float keep = upper ? p[k + half] : p[k];
            p[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (; off > 0; off /= 2) p[0] += __shfl_xor_sync(0xffffffffu, p[0], off);
    return p[0];
}

// WARPS per CTA, W of them per row, C columns per lane, RB rows at a time.
template <int WARPS, int W, int C, int RB, bool GRAD>
__global__ void __launch_bounds__(32 * WARPS, 1)
ls_pass_kernel(const __grid_constant__ PassArgs a) {
    constexpr bool MULTI = W > 1;
    constexpr int THREADS = 32 * WARPS, GROUPS = WARPS / W;
    grid_trigger();
    extern __shared__ __align__(16) unsigned char pass_smem[];
    __shared__ __align__(8) uint64_t bars[WARPS * kPassMaxSlots];
    __shared__ float red[2][RB][WARPS];
    __shared__ float xch[2][RB][WARPS * kPassMaxCluster];         // [parity][row][group][CTA][warp of the group]
    __shared__ __align__(8) uint64_t xch_bars[2][WARPS];          // [row parity][group]
    __shared__ double loss_sums[WARPS];
    __shared__ int last_issued[WARPS];                            // [group] chunk copied last
    __shared__ volatile int gave_up;                              // a wait ran out

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int grp = warp / W, wg = warp % W;
    const bool leader = wg == 0 && lane == 0;
    const uint32_t rank = MULTI && a.cluster > 1 ? cluster_rank() : 0u;
    const int64_t unit = MULTI && a.cluster > 1 ? blockIdx.x / a.cluster : blockIdx.x;
    const int64_t col0 = (int64_t)rank * a.slice;
    const int dn = (int)min((int64_t)a.slice, a.d - col0);
    const UnitRows owned = unit_rows(a.total, a.units, unit, a.d);
    const int64_t lo = owned.lo;
    const int nrows = owned.count;                                 // rows are counted from the unit's first
    const bool edge = owned.edge;
    const int R = a.chunk_rows;
    const int chunks = (nrows + R - 1) / R;
    int copied = rank == 0 ? min(chunks, a.hold_back) : chunks;    // chunks the leaders copy: all, but for a test, until a wait runs out
    const uint32_t row_bytes = (uint32_t)a.d * 4;
    const uint32_t ring = smem_u32(pass_smem) + a.ring_offset + (uint32_t)grp * a.slots * a.slot_bytes;
    const uint32_t bar0 = smem_u32(bars) + 8u * grp * a.slots;
    float *const flush = reinterpret_cast<float *>(pass_smem);
    if (tid == 0) gave_up = 0;
    if (leader) {
        last_issued[grp] = grp - GROUPS;
        for (int s = 0; s < a.slots; ++s) mbar_init(bar0 + 8 * s, 1);
        for (int f = 0; f < 2; ++f) mbar_init(smem_u32(&xch_bars[f][grp]), 1);
        fence_barrier_init();
    }

    // Copies of the leader: chunk after chunk of its group.  `src` is the first byte of the next one's rows.
    auto first_row = [&](int k) { return (a.reverse ? chunks - 1 - k : k) * R; };
    const uintptr_t unit_base = reinterpret_cast<uintptr_t>(a.A) + (uintptr_t)(lo * a.d + col0) * 4;
    const int64_t src_step = (a.reverse ? -(int64_t)GROUPS : (int64_t)GROUPS) * R * row_bytes;
    uintptr_t src = unit_base + (uint64_t)(uint32_t)max(first_row(grp), 0) * row_bytes;
    const uint64_t policy = l2_evict_first();
    auto issue = [&](int k, int s) {
        const uint32_t bar = bar0 + 8 * s;
        // the bytes [from, to) of A to shared memory, `from` going to `dst` (which agrees with it modulo 16)
        auto copy = [&](uintptr_t from, uintptr_t to, uint32_t dst) {
            const uint32_t origin = dst - (uint32_t)from;             // of address zero, so to say
            BulkRange r = bulk_range(from, to);
            if (edge) {
                const uintptr_t a_begin = reinterpret_cast<uintptr_t>(a.A);
                r = bulk_range_inside(r, a_begin, a_begin + (uintptr_t)(a.total * a.d) * 4);
                for (uintptr_t p = from; p < r.b0 && p < to; p += 4) store_shared(origin + (uint32_t)p, *reinterpret_cast<const float *>(p));
                for (uintptr_t p = r.b1 > from ? r.b1 : from; p < to; p += 4) store_shared(origin + (uint32_t)p, *reinterpret_cast<const float *>(p));
            }
            if (r.b1 > r.b0) {
                mbar_expect(bar, (uint32_t)(r.b1 - r.b0));
                bulk_copy(origin + (uint32_t)r.b0, reinterpret_cast<const void *>(r.b0), (uint32_t)(r.b1 - r.b0), bar, policy);
            }
        };
        const int count = min(R, nrows - first_row(k));
        const uint32_t dst = ring + (uint32_t)s * a.slot_bytes + (uint32_t)(src & 15);
        if (MULTI && a.cluster > 1)                     // a slice of each row
            for (int i = 0; i < count; ++i) {
                const uintptr_t from = src + (uintptr_t)((uint32_t)i * row_bytes);
                copy(from, from + (uint32_t)dn * 4, dst + (uint32_t)i * a.row_stride);
            }
        else
            copy(src, src + (uint32_t)count * row_bytes, dst);
        mbar_arrive(bar);
        src += src_step;
        last_issued[grp] = k;
    };
    constexpr int stride = 32 * W, CB = C < 4 ? C : 4;             // CB columns are tested for together
    const int first = lane + 32 * wg;
    // The first rows on their way to L2 while the kernels before this one finish (to L2 only: whoever still writes A writes
    // it there)
    if (leader && !edge && a.cluster == 1)
        for (int s = 0; s < a.slots; ++s) {
            const int k = grp + s * GROUPS;
            if (k >= chunks) break;
            const BulkRange r = prefetch_range(src + (int64_t)s * src_step, (uint32_t)min(R, nrows - first_row(k)) * row_bytes);
            if (r.b1 > r.b0) bulk_prefetch(reinterpret_cast<const void *>(r.b0), (uint32_t)(r.b1 - r.b0));
        }
    if constexpr (W == 16)                              // (the only ones in clusters, a slice of each row)
        if (leader && !edge && a.cluster > 1)
            for (int k = 0; k < min(a.slots, chunks); ++k)
                for (int i = 0; i < min(R, nrows - first_row(k)); ++i) {
                    const BulkRange r = prefetch_range(src + (int64_t)k * src_step + (int64_t)((uint32_t)i * row_bytes), (uint32_t)dn * 4);
                    if (r.b1 > r.b0) bulk_prefetch(reinterpret_cast<const void *>(r.b0), (uint32_t)(r.b1 - r.b0));
                }
    grid_wait();
    if (leader)
        for (int s = 0; s < a.slots; ++s)
            if (grp + s * GROUPS < copied) issue(grp + s * GROUPS, s);

    float xv[C], acc[GRAD ? C : 1];
#pragma unroll
    for (int c = 0; c < C; ++c) xv[c] = first + stride * c < dn ? __ldcg(a.x + col0 + first + stride * c) : 0.f;
    if (a.x_prev) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const float old = first + stride * c < dn ? __ldcg(a.x_prev + col0 + first + stride * c) : 0.f;
            xv[c] = fmaf(a.gamma, xv[c] - old, xv[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < (GRAD ? C : 1); ++c) acc[c] = 0.f;
    double loss = 0.0;
    __syncthreads();                                    // barriers initialised, for every warp of a group
    if (MULTI && a.cluster > 1) cluster_sync();         // and every CTA of the cluster has started

    // A wait that runs out ends its warp's part (lane by lane): it waits for nothing more, its leader copies nothing more, it
    // sends nothing to the cluster (whose other warps then run out of time in turn), and the CTA's results become NaN, so
    // that no wrong gradient or loss passes for a right one.  It goes on through its rows all the same, because the
    // barriers it shares with other warps count it.  (Each of these conditions is on the path of every chunk or row: a test of
    // `alive` before the refill in place of `copied`, or state kept in shared memory, cost 2 to 10 %.)
    bool alive = true;
    int flip = 0, xch_parity = 0;
    auto give_up = [&](int code) {
        alive = false;
        copied = 0;
        gave_up = 1;
        atomicMax(&g_pass_status, code);
    };

    // RBX rows whose first one starts at shared-memory address `at`, right-hand side bv in the lanes that get its sum.
    auto process = [&](auto batch, uint32_t at, float bv) {
        constexpr int RBX = decltype(batch)::value;
        float v[RBX][C];
        float2 s[RBX];
#pragma unroll
        for (int i = 0; i < RBX; ++i) s[i] = make_float2(0.f, 0.f);
        // All loads before the first multiply-add: were they in the same guarded block, every block would wait for its
        // own loads.  Columns four at a time: all lanes have them, or none, or some (those without read the row's last
        // columns and multiply them by the zeros in xv).
#pragma unroll
        for (int c0 = 0; c0 < C; c0 += CB) {
            if (stride * (c0 + CB) <= dn) {
#pragma unroll
                for (int i = 0; i < RBX; ++i)
#pragma unroll
                    for (int c = c0; c < c0 + CB; ++c)
                        v[i][c] = load_shared(at + (uint32_t)i * a.row_stride + 4u * (uint32_t)(first + stride * c));
            } else if (c0 == 0 || stride * c0 < dn) {
#pragma unroll
                for (int c = c0; c < c0 + CB; ++c) {
                    const uint32_t off = at + 4u * (uint32_t)min(first + stride * c, dn - 1);
#pragma unroll
                    for (int i = 0; i < RBX; ++i) v[i][c] = load_shared(off + (uint32_t)i * a.row_stride);
                }
            } else {
#pragma unroll
                for (int i = 0; i < RBX; ++i)
#pragma unroll
                    for (int c = c0; c < c0 + CB; ++c) v[i][c] = 0.f;
            }
        }
#pragma unroll
        for (int i = 0; i < RBX; ++i) {
            if constexpr (C == 1) {
                s[i].x = v[i][0] * xv[0];
            } else {
#pragma unroll
                for (int c = 0; c < C; c += 2)
                    s[i] = __ffma2_rn(make_float2(v[i][c], v[i][c + 1]), make_float2(xv[c], xv[c + 1]), s[i]);
            }
        }
        float p[RBX];
#pragma unroll
        for (int i = 0; i < RBX; ++i) p[i] = s[i].x + s[i].y;
        float dot = butterfly<RBX>(p, lane);
        constexpr int SHARE = 32 / RBX;                 // lanes that hold the sum of one row
        if constexpr (MULTI) {
            const int mine = lane / SHARE, sub = lane % SHARE;
            if (a.cluster > 1) {
                const int parts = W * a.cluster;                      // shares of a dot product
                const uint32_t bar = smem_u32(&xch_bars[flip][grp]);
                float *const share = &xch[flip][mine][grp * parts];
                if (leader && alive) mbar_arrive_expect(bar, 4u * parts * RBX);
                if (sub < a.cluster && alive) send_remote(smem_u32(share + rank * W + wg), bar, (uint32_t)sub, dot);
                if (alive && !mbar_wait(bar, xch_parity)) give_up(22);
                __syncwarp();
                dot = 0.f;
                for (int q = sub; q < parts; q += SHARE) dot += share[q];
                xch_parity ^= flip;
            } else {
                if (sub == 0) red[flip][mine][warp] = dot;
                __syncwarp();
                bar_sync(1 + grp, 32 * W);
                dot = sub < W ? red[flip][mine][grp * W + sub] : 0.f;
            }
#pragma unroll
            for (int o = SHARE / 2; o > 0; o /= 2) dot += __shfl_xor_sync(0xffffffffu, dot, o);
            flip ^= 1;
        }
        const float res = dot - bv;
        if constexpr (GRAD) {
#pragma unroll
            for (int i = 0; i < RBX; ++i) {
                const float ri = RBX == 1 ? res : __shfl_sync(0xffffffffu, res, i * SHARE);
                if constexpr (C == 1) {
                    acc[0] = fmaf(v[i][0], ri, acc[0]);
                } else {
#pragma unroll
                    for (int c = 0; c < C; c += 2) {
                        const float2 t = __ffma2_rn(make_float2(v[i][c], v[i][c + 1]), make_float2(ri, ri), make_float2(acc[c], acc[c + 1]));
                        acc[c] = t.x;
                        acc[c + 1] = t.y;
                    }
                }
            }
        } else {
            if (wg == 0 && lane % SHARE == 0) loss += (double)res * (double)res;
        }
    };

    bool loaded = false;
    int slot = 0, parity = 0;
    int k = grp;
    int row = first_row(k);
    // right-hand sides of the current chunk (lane l: its row l) and of the next one, fetched a chunk ahead
    const float *const rhs = a.b + lo;
    auto fetch_rhs = [&](int chunk) {
        if (chunk >= chunks) return 0.f;
        const int r = first_row(chunk) + lane;
        return lane < R && r < nrows ? __ldcg(rhs + r) : 0.f;
    };
    float b_now = fetch_rhs(k), b_next = fetch_rhs(k + GROUPS);
    int64_t machine = GRAD ? lo / a.rows : 0;
    int seg_end = GRAD ? (int)min((int64_t)nrows, (machine + 1) * a.rows - lo) : nrows;
    for (;;) {
        while (k < chunks && row < seg_end) {
            const int r0 = first_row(k), r1 = min(r0 + R, nrows);
            if (!loaded) {
                if (alive && !mbar_wait(bar0 + 8 * slot, parity)) give_up(21);
                loaded = true;
            }
            const uint32_t mis = ((uint32_t)unit_base + (uint32_t)r0 * row_bytes) & 15;
            const uint32_t chunk_at = ring + (uint32_t)slot * a.slot_bytes + mis;
            const int stop = min(r1, seg_end);          // the rest of the chunk belongs to the next machine
            using batch_rows = std::integral_constant<int, RB>;
            using single_row = std::integral_constant<int, 1>;
            for (; row + RB <= stop; row += RB)
                process(batch_rows{}, chunk_at + (uint32_t)(row - r0) * a.row_stride,
                        __shfl_sync(0xffffffffu, b_now, (row - r0 + lane / (32 / RB)) & 31));
            if constexpr (RB > 1)
                for (; row < stop; ++row)
                    process(single_row{}, chunk_at + (uint32_t)(row - r0) * a.row_stride,
                            __shfl_sync(0xffffffffu, b_now, (row - r0) & 31));
            row = stop;
            if (stop == r1) {                           // the chunk is used up
                // every warp of the group has read its part of the rows (in a cluster and between warps the exchange of
                // the last row's shares told so): the slot may be refilled
                __syncwarp();
                if (leader && k + a.slots * GROUPS < copied) issue(k + a.slots * GROUPS, slot);
                k += GROUPS;
                b_now = b_next;
                b_next = fetch_rhs(k + GROUPS);
                loaded = false;
                if (k < chunks) row = first_row(k);
                if (++slot == a.slots) { slot = 0; parity ^= 1; }
            }
        }
        if constexpr (GRAD) {
            // partial gradient of this unit for this machine
            const int64_t machine_unit = (machine * a.rows + 1) * a.units - 1;      // unit of the machine's first row
            float *out = a.part + (machine * a.slots_per_machine + (unit - machine_unit / a.total)) * a.ldp + col0;
            auto each_column = [&](auto &&f) {
#pragma unroll
                for (int c = 0; c < C; ++c)
                    if (first + stride * c < dn) f(c, first + stride * c);
            };
            if constexpr (GROUPS == 1) {
                each_column([&](int c, int col) { out[col] = acc[c]; });
            } else {
                __syncthreads();                        // where it is the rings that take the groups' sums
                const int room = min(a.flush_floats / dn, GROUPS);
                for (int g0 = 0; g0 < GROUPS; g0 += room) {           // as many groups at a time as there is room for
                    if (grp >= g0 && grp < g0 + room) each_column([&](int c, int col) { flush[(grp - g0) * dn + col] = acc[c]; });
                    __syncthreads();
                    const int here = min(room, GROUPS - g0);
                    for (int col = tid; col < dn; col += THREADS) {
                        float sum = g0 > 0 ? out[col] : 0.f;
#pragma unroll 4
                        for (int g = 0; g < here; ++g) sum += flush[g * dn + col];
                        out[col] = sum;
                    }
                    __syncthreads();
                }
            }
            if (gave_up) {                              // (threads overwrite what they wrote themselves)
                if constexpr (GROUPS == 1) {
#pragma unroll 1
                    for (int col = first; col < dn; col += stride) out[col] = __int_as_float(0x7fffffff);
                } else
#pragma unroll 1
                    for (int col = tid; col < dn; col += THREADS) out[col] = __int_as_float(0x7fffffff);
            }
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] = 0.f;
        }
        if (seg_end == nrows) break;
        ++machine;
        seg_end = (int)min((int64_t)nrows, seg_end + a.rows);
    }
    if constexpr (!GRAD) {
#pragma unroll
        for (int o = 16; o > 0; o /= 2) loss += __shfl_xor_sync(0xffffffffu, loss, o);
        if (lane == 0) loss_sums[warp] = loss;
        __syncthreads();
        if (tid == 0 && rank == 0) {
            double sum = 0.0;
            for (int w = 0; w < WARPS; ++w) sum += loss_sums[w];
            a.loss_part[unit] = gave_up ? __longlong_as_double(0x7fffffffffffffffll) : sum;
        }
    }
    if (leader && !alive) {
        // Copies in flight must not outlive the CTA's shared memory: the last ones issued, one per slot at most (the i-th
        // went to slot i % slots and completes its phase i / slots).
        const int issued = (last_issued[grp] - grp) / GROUPS + 1;
        for (int i = max(issued - a.slots, 0); i < issued; ++i) mbar_wait(bar0 + 8 * (i % a.slots), (i / a.slots) & 1);
    }
    if (MULTI && a.cluster > 1) {
        cluster_sync();                                 // a CTA stays while others may still send to it
        if (!alive)                                     // ... and until what nobody waited for has arrived
            for (int i = 0; i < 100; ++i) __nanosleep(1000);
    }
}

// G[i][k] = inv_rows * sum of machine i's partial gradients, in the order of its units.  *clear = 0 (where it is not null) for a
// later kernel of the step.
__global__ void ls_pass_reduce_kernel(const float *__restrict__ part, int64_t rows, int64_t total, int64_t units,
                                      int slots_per_machine, int64_t ldp, int64_t d, float inv_rows, float *__restrict__ G, float *clear) {
    grid_trigger();
    grid_wait();
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0.f;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = blockIdx.y;
    if (k >= d) return;
    const int64_t first = ((i * rows + 1) * units - 1) / total, last = ((i + 1) * rows * units - 1) / total;
    const float *p = part + i * slots_per_machine * ldp + k;
    G[i * d + k] = sum_strided<16>(p, (int)(last - first) + 1, ldp) * inv_rows;
}

// loss[0] = scale * sum of the units' sums of squares: lane l sums units l, l + 32, ..., then a fixed tree.
__global__ void ls_loss_sum_kernel(const double *__restrict__ loss_part, int64_t units, double scale, double *loss) {
    grid_trigger();
    grid_wait();
    double s = sum_strided<8>(loss_part + threadIdx.x, (int)((units - threadIdx.x + 31) / 32), 32);
#pragma unroll
    for (int o = 16; o > 0; o /= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) loss[0] = s * scale;
}

cudaError_t launch_pass(const LsPass &p, PassArgs &a, const float *A, const float *b, const LsPoint &at, int64_t d,
                        cudaStream_t stream) {
    const bool grad = a.part != nullptr;
    a.A = A;
    a.b = b;
    a.x = at.x;
    a.x_prev = at.x_prev;
    a.gamma = at.gamma;
    a.d = d;
    a.rows = p.rows;
    a.total = p.total;
    a.units = p.units;
    a.ldp = p.ldp;
    a.slots_per_machine = p.slots_per_machine;
    a.cluster = p.cluster;
    a.slice = p.slice;
    a.chunk_rows = p.chunk_rows;
    a.slots = p.slots;
    a.hold_back = p.hold_back;
    a.slot_bytes = p.slot_bytes;
    a.row_stride = p.row_stride;
    a.ring_offset = p.ring_offset;
    a.flush_floats = (int)((p.ring_offset ? p.ring_offset : p.smem) / sizeof(float));
    auto go = [&](auto kernel) {
        if (cudaError_t e = allow_shared(reinterpret_cast<const void *>(kernel), p.smem)) return e;
        const ChainedLaunch launch(true, dim3((unsigned)(p.units * p.cluster)), dim3((unsigned)(32 * p.warps)), p.smem, stream, p.cluster);
        return cudaLaunchKernelEx(&launch.cfg, kernel, a);
    };
    auto pick = [&](auto warps, auto per_row, auto columns) {
        constexpr int WARPS = decltype(warps)::value, W = decltype(per_row)::value, C = decltype(columns)::value;
        constexpr int RB = pass_batch(W, C);
        return grad ? go(ls_pass_kernel<WARPS, W, C, RB, true>) : go(ls_pass_kernel<WARPS, W, C, RB, false>);
    };
    using std::integral_constant;
    using i1 = integral_constant<int, 1>;
    using i2 = integral_constant<int, 2>;
    using i4 = integral_constant<int, 4>;
    using i8 = integral_constant<int, 8>;
    using i12 = integral_constant<int, 12>;
    using i16 = integral_constant<int, 16>;
    using i20 = integral_constant<int, 20>;
    using i24 = integral_constant<int, 24>;
    using i28 = integral_constant<int, 28>;
    using i32 = integral_constant<int, 32>;
    auto wide = [&](auto warps, auto per_row) {
        constexpr int W = decltype(per_row)::value;
        if constexpr (W == 2)
            if (p.columns == 12) return pick(i16{}, per_row, i12{});
        if constexpr (W < 16)
            if (p.columns == 16) return pick(warps, per_row, i16{});
        if (p.columns == 20) return pick(warps, per_row, i20{});
        if constexpr (W == 16)
            if (p.columns == 28) return pick(warps, per_row, i28{});
        if constexpr (W >= 8)
            if (p.columns == 32) return pick(warps, per_row, i32{});
        return pick(warps, per_row, i24{});
    };
    switch (p.group_warps) {
        case 16: return wide(i16{}, i16{});
        case 8: return wide(i8{}, i8{});
        case 4: return wide(i8{}, i4{});
        case 2: return wide(i8{}, i2{});
        default: break;
    }
    switch (p.columns) {
        case 1: return pick(i16{}, i1{}, i1{});
        case 2: return pick(i16{}, i1{}, i2{});
        case 4: return pick(i16{}, i1{}, i4{});
        case 8: return pick(i16{}, i1{}, i8{});
        default: return pick(i16{}, i1{}, i16{});
    }
}

}  // namespace

LsPass make_ls_pass(int32_t n, int64_t rows, int64_t d, bool machines_apart, int sm_count) {
    LsPass p{};
    if (d > (int64_t)kPassCtaCols * kPassMaxCluster) return p;             // units == 0: does not apply
    p.cluster = 1;
    while (d > (int64_t)kPassCtaCols * p.cluster) p.cluster *= 2;
    p.slice = p.cluster == 1 ? (int)d : (int)(((d + p.cluster - 1) / p.cluster + 3) / 4 * 4);
    p.group_warps = 1;
    // (16 warps with 20 columns per lane instead of 24 where they suffice, us: 16 x 256 rows of 20000: 72.5 -> 70.5, 16 x 512 of
    // 8200: 53.2 -> 50.6.)  24 columns per lane at most where several warps share a row (four rows at a time, see pass_batch), 32 where that is
    // more than 8 warps hold.  One warp with 32 columns per lane handled one row at a time: from 513 columns two warps
    // with four rows are faster (gradients, 50 x 1200 rows of 600: 44 -> 29 us, of 1000: 48 -> 44).  Up to 12 columns
    // per lane 16 warps per CTA have the registers for that (37 with 8); with fewer columns per lane and more warps
    // per row than this, longer rows were slower (784: 41 -> 46, 6100: equal).
    if (p.slice > kPassOneWarp)
        do p.group_warps *= 2;
        while (p.group_warps < 8 && p.slice > 768 * p.group_warps);
    if (p.slice > 1024 * p.group_warps) p.group_warps = kPassMaxWarps;
    const int per_lane = (p.slice + 32 * p.group_warps - 1) / (32 * p.group_warps);
    p.columns = 1;
    while (p.columns < per_lane) p.columns *= 2;
    if (p.group_warps > 1) p.columns = per_lane > 20 ? (per_lane + 3) / 4 * 4 : per_lane > 16 || p.group_warps == kPassMaxWarps ? 20 : per_lane > 12 ? 16 : 12;
    const uint32_t smem = 220u * 1024u;
    if (p.columns == 28) {
        // Two rows at a time want room for two slots of two rows, and rows enough per unit (before that the ring's start, in chunks of two
        // rows, counts more than the chain).  us, one row at a time -> two, by rows per unit: one CTA per row (13300 columns), 4: 21.0 ->
        // 23.7, 16: 5 % slower, 24: equal, 40: 4 % faster; clusters of two (26476), 4: 26.7 -> 28.6, 8 to 11: 1 to 4 % faster, 16: 2 % slower,
        // 24: 3 % faster; of four and eight, 2: 1 to 2 % slower, 3: 4 % faster, 8: 8 to 11 %.
        const int64_t least = p.cluster == 1 ? 24 : p.cluster == 2 ? 8 : 3;
        if (p.group_warps < kPassMaxWarps || 4 * (p.slice * 4 + 56) > (int)smem || (int64_t)n * rows * p.cluster < least * sm_count) p.columns = 32;
    }
    p.warps = p.group_warps == 1 || p.columns == 12 || p.group_warps == 16 ? 16 : 8;
    const int groups = p.warps / p.group_warps;
    const uint32_t row_bytes = (uint32_t)p.slice * 4;
    const int batch = pass_batch(p.group_warps, p.columns);               // rows at a time
    p.chunk_rows = batch;
    if (p.group_warps == 1) p.chunk_rows *= std::max(1, std::min((int)(kPassRingBytes / (3 * groups) / (row_bytes * batch)), 32 / batch));
    p.row_stride = p.cluster == 1 ? row_bytes : (row_bytes + 31) / 16 * 16 + (uint32_t)(d * 4 % 16);
    p.slot_bytes = (p.chunk_rows * p.row_stride + 12 + 15) / 16 * 16;
    // half the room for the groups' sums (still one group's) where that makes the difference to a second ring slot
    const uint32_t all = (uint32_t)groups * p.slot_bytes;
    p.ring_offset = !machines_apart || groups == 1 ? 0u : kPassFlushBytes + 2 * all <= smem ? kPassFlushBytes : kPassFlushBytes / 2;
    const int room = (int)((smem - p.ring_offset) / all);
    p.slots = std::max((int)(kPassRingBytes / (groups * p.slot_bytes)), 3);
    p.slots = std::min({p.slots, room, kPassMaxSlots});
    if (p.slots < 2) return LsPass{};
    p.smem = p.ring_offset + (size_t)groups * p.slots * p.slot_bytes;
    p.total = (int64_t)n * rows;
    p.rows = machines_apart ? rows : p.total;
    p.units = sm_count / p.cluster;
    if (p.cluster > 1) {
        // no more clusters than run side by side: SMs that cannot form another one stay idle, a second wave would cost more
        auto kernel = ls_pass_kernel<16, 16, 32, 1, true>;
        int resident = 0;
        ChainedLaunch launch(true, dim3((unsigned)(p.units * p.cluster)), dim3((unsigned)(32 * p.warps)), p.smem, nullptr, p.cluster);
        launch.cfg.attrs = &launch.attrs[1];                               // the cluster's size alone
        launch.cfg.numAttrs = 1;
        if (allow_shared(reinterpret_cast<const void *>(kernel), p.smem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&resident, kernel, &launch.cfg) != cudaSuccess || resident < 1) {
            cudaGetLastError();
            return LsPass{};
        }
        if (p.units > resident) p.units = resident;
    }
    if (p.units > p.total) p.units = p.total;
    p.ldp = (d + 3) / 4 * 4;
    p.slots_per_machine = 1;
    const int64_t machines = p.total / p.rows;
    for (int64_t i = 0; i < machines; ++i) {
        const int64_t first = ((i * p.rows + 1) * p.units - 1) / p.total, last = ((i + 1) * p.rows * p.units - 1) / p.total;
        if (last - first + 1 > p.slots_per_machine) p.slots_per_machine = (int)(last - first + 1);
    }
    return p;
}

size_t ls_pass_partials(const LsPass &p) { return p.units ? (size_t)(p.total / p.rows) * p.slots_per_machine * p.ldp : 0; }

cudaError_t launch_ls_pass_gradients(const LsPass &p, const float *A, const float *b, const LsPoint &at, int64_t d,
                                     float *part, cudaStream_t stream) {
    PassArgs a{};
    a.part = part;
    return launch_pass(p, a, A, b, at, d, stream);
}

cudaError_t launch_ls_pass_loss(const LsPass &p, const float *A, const float *b, const LsPoint &at, int64_t d, bool reverse,
                                double *loss_part, cudaStream_t stream) {
    PassArgs a{};
    a.loss_part = loss_part;
    a.reverse = reverse;
    return launch_pass(p, a, A, b, at, d, stream);
}

cudaError_t launch_ls_pass_reduce(const LsPass &p, const float *part, int64_t d, float inv_rows, float *G, float *clear, cudaStream_t stream) {
    const int n = (int)(p.total / p.rows);
    return launch_chained(true, ls_pass_reduce_kernel, dim3((unsigned)((d + 127) / 128), n), dim3(128), 0, stream, part, p.rows, p.total, p.units,
                          p.slots_per_machine, p.ldp, d, inv_rows, G, clear);
}

cudaError_t launch_ls_loss_sum(const double *loss_part, int64_t units, double scale, double *loss, cudaStream_t stream) {
    return launch_chained(true, ls_loss_sum_kernel, dim3(1), dim3(32), 0, stream, loss_part, units, scale, loss);
}

// Host-side replay of the copies and prefetches of one pass over a matrix at address `a_begin`.
void ls_pass_reads(const LsPass &p, int64_t d, uintptr_t a_begin, int64_t *before, int64_t *behind) {
    const uintptr_t a_end = a_begin + (uintptr_t)(p.total * d) * 4;
    const uint32_t row_bytes = (uint32_t)d * 4;
    *before = *behind = 0;
    auto touch = [&](BulkRange r) {
        if (r.b1 <= r.b0) return;
        if (r.b0 < a_begin) *before = std::max(*before, (int64_t)(a_begin - r.b0));
        if (r.b1 > a_end) *behind = std::max(*behind, (int64_t)(r.b1 - a_end));
    };
    for (int64_t unit = 0; unit < p.units; ++unit) {
        const UnitRows u = unit_rows(p.total, p.units, unit, d);
        auto copy = [&](uintptr_t from, uintptr_t to) {
            const BulkRange r = bulk_range(from, to);
            touch(u.edge ? bulk_range_inside(r, a_begin, a_end) : r);
        };
        for (int row = 0; row < u.count; row += p.chunk_rows) {
            const int count = std::min(p.chunk_rows, u.count - row);
            const uintptr_t src = a_begin + (uintptr_t)((u.lo + row) * d) * 4;
            if (p.cluster == 1) {
                copy(src, src + (uint32_t)count * row_bytes);
                if (!u.edge) touch(prefetch_range(src, (uint32_t)count * row_bytes));
                continue;
            }
            for (int i = 0; i < count; ++i)
                for (int64_t col = 0; col < d; col += p.slice) {
                    const uintptr_t from = src + (uintptr_t)i * row_bytes + (uintptr_t)col * 4;
                    const uint32_t bytes = (uint32_t)std::min<int64_t>(p.slice, d - col) * 4;
                    copy(from, from + bytes);
                    if (!u.edge) touch(prefetch_range(from, bytes));
                }
        }
    }
}

cudaError_t ls_pass_take_status(int *status) {
    cudaError_t e = cudaMemcpyFromSymbol(status, g_pass_status, sizeof(int));
    if (e != cudaSuccess || *status == 0) return e;
    const int zero = 0;
    return cudaMemcpyToSymbol(g_pass_status, &zero, sizeof(int));
}

}  // namespace core
