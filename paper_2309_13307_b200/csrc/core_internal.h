// Internal declarations shared by the translation units of the CORE library.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "core_rng.cuh"

namespace core {

// Grants `kernel` that much dynamic shared memory on the current device (once; later calls only look it up).
cudaError_t allow_shared(const void *kernel, size_t bytes);

// Launches a kernel of a chain: it may be scheduled while its predecessor in the stream drains (programmatic stream
// serialisation), which hides its launch latency (1 to 1.5 us a kernel).  Such a kernel calls grid_wait() before it touches
// global memory: what every earlier kernel of the stream wrote is then visible to its ordinary loads, cached in L1 or not.  It
// is not to the read-only path, so no __ldg there, and no plain reads through `const T *__restrict__`, which the compiler
// may turn into such loads: __ldcg, or pointers without __restrict__.
struct ChainedLaunch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attrs[2];
    ChainedLaunch(bool chain, dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int cluster = 1) {
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[0].val.programmaticStreamSerializationAllowed = chain ? 1 : 0;
        attrs[1].id = cudaLaunchAttributeClusterDimension;
        attrs[1].val.clusterDim.x = (unsigned)cluster;
        attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
        cfg.attrs = attrs;
        cfg.numAttrs = cluster > 1 ? 2 : 1;
    }
};
template <typename... P, typename... A>
cudaError_t launch_chained(bool chain, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
    if (cudaError_t e = allow_shared(reinterpret_cast<const void *>(kernel), smem)) return e;
    const ChainedLaunch launch(chain, grid, block, smem, stream);
    return cudaLaunchKernelEx(&launch.cfg, kernel, static_cast<P>(args)...);
}
// CTAs of a chained kernel go wherever there is room first.  If they do not fill the chip, that packs them on few SMs (n = 7,
// d = 3210, m = 940: 45 -> 64 us), so kernels that generate are chained only where they do fill it (`capacity` CTAs are
// resident together), or where the whole work, d * m Gaussians, takes less than the 2 us or so that are at stake.
inline bool chain_pays(int64_t ctas, int64_t capacity, int64_t d, int64_t m) {
    return ctas * 10 >= capacity * 9 || d <= ((int64_t)1 << 21) / m;
}

constexpr int kThreads = 256;        // threads per CTA in the round kernels
constexpr int kMaxGroup = 16;        // machines handled by one pass of the scalar projection
constexpr int kMaxGroupTc = 64;      // most machines one pass of the tensor-memory projection can take

// Machines the next projection pass takes when n_left remain: up to 64 (32 where a CTA holds one group of
// 128 vectors only) where the tensor-memory kernel applies to more than 16, otherwise at most 16.
int32_t project_group(int32_t n_left, int32_t m);
// Test hook: -1 = choose by shape (default); 0 or 1 = always the scalar kernel; 2 = the tensor-memory kernel for any group
// of machines it can take.
void project_force_kernel(int kind);
bool project_kernel_forced();      // anything but -1

// Launch geometry of one projection pass, fixed by (n, m, d, dtype) on the host.
struct ProjectPlan {
    int nb;           // machines per pass rounded up to 1, 2, 4, 8 or 16
    int jt;           // vectors per thread
    int uq;           // coordinate blocks per thread per step
    int tile_q;       // coordinate blocks (of 4) per shared-memory tile
    int tj;           // threads across vectors (power of two)
    int tq;           // threads across coordinate blocks = kThreads / tj
    int grid_x;       // CTAs across coordinates
    int grid_y;       // CTAs across vectors
    int64_t tiles;    // ceil(d / (4 * tile_q))
    size_t smem;      // dynamic shared memory per CTA
    bool tc;          // the tcgen05 kernel
    bool chain;       // see chain_pays
};

ProjectPlan make_project_plan(int32_t n_group, int32_t m, int64_t d, int dtype, int sm_count);

// tcgen05 variant (core_project_tc.cu): 128 or 256 vectors per CTA, up to project_tc_max_group(m) machines per
// pass (N = 16, 32 or 64 of the instruction), accumulators in tensor memory; same partial-sum layout.  q_base must be a multiple of 64 blocks.  Its waits are bounded: a wait that
// runs out raises a device status word, which project_tc_take_status returns and clears after
// synchronising the device.
bool project_tc_applies(int32_t n_group, int32_t m);
int32_t project_tc_max_group(int32_t m);   // 64 with 256 vectors per CTA, otherwise 32
void fill_project_tc_plan(ProjectPlan &plan, int32_t n_group, int32_t m, int64_t d, int dtype, int sm_count);
cudaError_t launch_project_tc(const ProjectPlan &plan, const RoundKeys &keys, uint32_t t, const void *G,
                              int dtype, int32_t n, int64_t ldg, int64_t d, int32_t m, uint64_t q_base,
                              float *partial, cudaStream_t stream);
cudaError_t project_tc_take_status(int *status);
// One small CTA that waits, with the projection's bounded-wait helper, on a barrier nobody completes:
// after limit_ns the wait gives up, the status word receives `code`, and observed_dev[0..1] (device)
// become {0: the wait did not succeed, 1: the second warp saw the abort flag}.
cudaError_t launch_wait_timeout_probe(uint64_t limit_ns, int code, uint32_t *observed_dev, cudaStream_t stream);

// One projection pass over coordinates [0, d) of rows G + i*ldg, i < n <= 16.
// q_base is the global index of the block holding coordinate 0 of G (non-zero when G
// is a slab of a longer vector).  Writes partial[(c * n + i) * m + j], c < plan.grid_x.
cudaError_t launch_project(const ProjectPlan &plan, const RoundKeys &keys, uint32_t t, const void *G,
                           int dtype, int32_t n, int64_t ldg, int64_t d, int32_t m, uint64_t q_base,
                           float *partial, cudaStream_t stream);

// Projection of one combined row (core_project_row.cu): partial[c*m + j] = the share of CTA column c in
// <scale * (row 0 + row 1 + ... + row rows-1), xi_j>.  Rows are `ldg` elements apart and of any alignment.
struct RowPlan {
    int tile_q;       // coordinate blocks (of 4) per shared-memory tile
    int tj;           // threads across vectors (four vectors each)
    int tq;           // threads across coordinate blocks
    int grid_x;       // CTAs across coordinates
    int grid_y;       // CTAs across vectors
    int compute;      // generating threads of a CTA
    int64_t tiles;
    size_t smem;
    bool chain;       // see chain_pays
    bool turn;        // angles from the table (core_rng.cuh)
};
RowPlan make_row_plan(const void *G, int dtype, int32_t rows, int64_t ldg, int32_t m, int64_t d, int sm_count);
int row_plan_columns(int32_t m, int64_t d, int sm_count);      // most CTA columns of any rows' plan
cudaError_t launch_project_row(const RowPlan &plan, const RoundKeys &keys, uint32_t t, const void *G, int dtype,
                               int32_t rows, int64_t ldg, float scale, int64_t d, int32_t m, uint64_t q_base,
                               float *partial, cudaStream_t stream);

// P[i*m+j] = (accumulate ? P[i*m+j] : 0) + sum_c partial[c][i][j], c ascending.
cudaError_t launch_finish_project(const float *partial, int chunks, int32_t n, int32_t m, float *P,
                                  bool accumulate, cudaStream_t stream);

// pbar[j] = (1/n) sum_i (sum_c partial[c][i][j]): finish + aggregate for one group of machines, same order.
cudaError_t launch_finish_aggregate(const float *partial, int chunks, int32_t n, int32_t m, float *pbar,
                                    cudaStream_t stream);

cudaError_t launch_aggregate(const float *P, int32_t n, int32_t m, float *pbar, cudaStream_t stream);

// out[k - k_begin] = gtilde[k] for k in [k_begin, k_end); k_begin must be a multiple of 2048.
// With an epilogue the estimate is consumed where it is produced and never stored:
//   out[k] = base[k] - step * gtilde[k]   (the optimiser update of Algorithms 2 and 4)
// and, if shift_dst is set, shift_dst[k] = shift_src[k] first (x_prev <- x of Algorithm 4).  With lookahead set the base is
// shift_src[k] + gamma * (shift_src[k] - shift_dst[k]), formed from the values before the shift, instead of base[k].
// out may alias base and shift_src; all four arrays are indexed like out.
// step_dev, when set, overrides step: the kernel reads the step from device memory (a step that an
// earlier kernel of the same iteration chose, as in Option I of Algorithm 3), times step_scale.
struct ReconstructEpilogue {
    const float *base;
    float step;
    const float *shift_src;
    float *shift_dst;
    const float *step_dev = nullptr;
    float step_scale = 1.0f;
    bool lookahead = false;
    float gamma = 0.f;
};
// With parts the message is not in pbar yet: the kernel forms it from the projection's partial sums (partial[c][i][j],
// c < chunks, i < n; the same bits as launch_finish_aggregate) and writes it there.  reconstruct_joins tells where it can.
struct MessageParts {
    const float *partial;
    int chunks;
    int n;
};
enum class RecKernel { kShort, kWide, kTurn };         // for short vectors; for long ones, without and with the table of angles
RecKernel reconstruct_kernel_for(int64_t nq, int32_t m, int sm_count);     // nq blocks of four coordinates
bool reconstruct_joins(int chunks, int32_t n, int32_t m, int64_t d, int sm_count);
cudaError_t launch_reconstruct(const RoundKeys &keys, uint32_t t, float *pbar, int32_t m,
                               int64_t k_begin, int64_t k_end, float *out, int sm_count,
                               cudaStream_t stream, const ReconstructEpilogue *epilogue = nullptr,
                               const MessageParts *parts = nullptr);

// The whole round of a short vector in one launch of one cluster (core_short.cu): `machines` messages of a row each (the very numbers
// of the separate kernels), or one message of the sum of `rows` rows times scale.  pbar receives the combined message.
struct ShortPlan {
    int ctas;         // of the cluster; 0: the kernel does not apply
    int per;          // blocks per CTA
    int stride;       // of the Gaussians' rows in shared memory, in blocks
    int lanes;        // threads that share a vector's projection
    int slices;       // ranges of the vectors in the reconstruction
    int columns, tile, tq, uq;       // several messages: columns, blocks and lanes of the separate kernel's tiles
    size_t smem;
};
// Test hook: none of these kernels.
void short_kernels_set(bool on);
bool short_kernels_off();
ShortPlan make_short_plan(int32_t machines, int32_t rows, int32_t m, int64_t d, int sm_count);
// The reconstruction alone, with the same bits (per and ctas of the plan do not matter): `per` blocks and `threads` threads per CTA.
struct ShortGrid {
    int per, threads, ctas;
};
ShortGrid make_short_grid(const ShortPlan &plan, int32_t m, int64_t d, int sm_count, const MessageParts *parts);
cudaError_t launch_short_reconstruct(const ShortPlan &plan, const RoundKeys &keys, uint32_t t, float *pbar, int64_t d, int32_t m, float *out,
                                     int sm_count, const ReconstructEpilogue *epilogue, const MessageParts *parts, cudaStream_t stream);
// With P not null (one message) it is written there and nothing is reconstructed.
cudaError_t launch_short_round(const ShortPlan &plan, const RoundKeys &keys, uint32_t t, const void *G, int dtype, int32_t rows,
                               int32_t machines, int64_t ldg, float scale, int64_t d, int32_t m, float *P, float *pbar, float *out,
                               const ReconstructEpilogue *epilogue, cudaStream_t stream);

cudaError_t launch_debug_philox(const RoundKeys &keys, uint32_t t, uint32_t j, uint64_t q0, int64_t nq,
                                uint32_t *words, cudaStream_t stream);
cudaError_t launch_debug_gaussians(const RoundKeys &keys, uint32_t t, uint32_t j, uint64_t q0, int64_t nq,
                                   float *z, cudaStream_t stream);
cudaError_t launch_debug_box_muller(const uint32_t *words, int64_t nb, float *z, cudaStream_t stream);

// Least squares.  Pass 1: res[i*rows + r] = A_i[r] . x - b_i[r].  Pass 2: the rows of a
// machine are cut into `splits` ranges; part[(i*splits + s)*d + k] = sum over the rows of
// range s of A_i[r][k] * res_i[r].  Reduce: G[i*d + k] = (1/rows) sum_s part[i][s][k].
struct LsPlan {
    int splits;
    int rows_per_split;
};
LsPlan make_ls_plan(int32_t n, int32_t rows, int64_t d, int sm_count);
cudaError_t launch_ls_residual(const float *A, const float *b, const float *x, int32_t n, int32_t rows,
                               int64_t d, float *res, cudaStream_t stream);
cudaError_t launch_ls_at_r(const LsPlan &plan, const float *A, const float *res, int32_t n, int32_t rows,
                           int64_t d, float *part, cudaStream_t stream);
cudaError_t launch_ls_reduce(const LsPlan &plan, const float *part, int32_t n, int32_t rows, int64_t d,
                             float *G, float *clear, cudaStream_t stream);
// Single pass over A (core_ls_pass.cu) for rows of up to 131072 columns of any alignment: the residual of each row is
// formed on the fly, A is read from HBM once.  The n * rows rows are cut over `units` CTAs (or clusters); a unit's
// partial gradient goes to part[(i * slots_per_machine + s) * ldp + k], s counting the units that hold rows of
// machine i, or, when the machines are not kept apart, to part[unit * ldp + k].
struct LsPass {
    int64_t units;            // 0: the kernel does not apply to this shape
    int64_t rows, total;      // rows per (kept-apart) machine, rows of all
    int64_t ldp;
    int slots_per_machine;
    int cluster, slice, warps, group_warps, columns, chunk_rows, slots;
    uint32_t slot_bytes, row_stride, ring_offset;
    size_t smem;
    int hold_back = INT32_MAX;   // test: chunks of rows from this one on are never copied, so that a wait runs out
};
struct LsPoint {              // x, or x + gamma (x - x_prev) (the look-ahead point of Algorithm 4)
    const float *x;
    const float *x_prev = nullptr;
    float gamma = 0.f;
};
LsPass make_ls_pass(int32_t n, int64_t rows, int64_t d, bool machines_apart, int sm_count);
size_t ls_pass_partials(const LsPass &pass);      // floats
cudaError_t launch_ls_pass_gradients(const LsPass &pass, const float *A, const float *b, const LsPoint &at, int64_t d,
                                     float *part, cudaStream_t stream);
cudaError_t launch_ls_pass_reduce(const LsPass &pass, const float *part, int64_t d, float inv_rows, float *G,
                                  float *clear, cudaStream_t stream);
// loss_part[u] = sum of squared residuals of unit u; with `reverse` from the last row to the first.
cudaError_t launch_ls_pass_loss(const LsPass &pass, const float *A, const float *b, const LsPoint &at, int64_t d, bool reverse,
                                double *loss_part, cudaStream_t stream);
cudaError_t launch_ls_loss_sum(const double *loss_part, int64_t units, double scale, double *loss, cudaStream_t stream);
// Bytes before and behind a matrix at address a_begin that the bulk copies and prefetches of a pass would touch (host only).
void ls_pass_reads(const LsPass &pass, int64_t d, uintptr_t a_begin, int64_t *before, int64_t *behind);
cudaError_t ls_pass_take_status(int *status);     // after a device synchronisation; clears the word
// Comparison step of Algorithm 3, on the device: if *f_trial < *f then x <- trial, *f <- *f_trial and the
// flag is 1, otherwise nothing changes and the flag is 0 (a tie keeps x).  f_trial is scale times the sum of the
// `parts` numbers f_parts.  flag_scratch is a device int owned by the caller of this function; flag_out (may be
// null) receives a copy.
cudaError_t launch_keep_better(const double *f_parts, int64_t parts, double scale, const float *trial, int64_t d, double *f,
                               float *x, int *flag_scratch, int32_t *flag_out, cudaStream_t stream);
// y = x + gamma (x - x_prev)
cudaError_t launch_lookahead(const float *x, const float *x_prev, float gamma, int64_t d, float *y, cudaStream_t stream);
// loss[0] = sum of res^2 over all rows of all machines, in double in a fixed order
cudaError_t launch_ls_loss(const float *res, int32_t n, int32_t rows, double *loss, cudaStream_t stream);

// Option I of Algorithm 3: p_out[0] (may be null) = sqrt((1/m) sum_j pbar_j^2), h_out[0] =
// min{ m / (16 r1), c H^-1/2 p^-1/2 d^-3/4 m^3/4 }, both formed on the device in double and stored as float.
cudaError_t launch_option1_step(const float *pbar, int32_t m, int64_t d, double r1, double H, double c, float *p_out,
                                float *h_out, cudaStream_t stream);
// Algorithm 5's averaging by gossip: out[i*m + j] = sum_l W[i*n + l] in[l*m + j], l ascending (in != out).
cudaError_t launch_gossip_round(const float *W, const float *in, int32_t n, int32_t m, float *out, cudaStream_t stream);
// What lies between the projection and the reconstruction of a decentralised step, for up to 64 machines (gossip_step_applies):
// out = W^rounds P, where P is given, or comes from the projection's partial sums partial[c][i][j], c < chunks (the bits of
// launch_finish_project; gossip_joins tells where that pays); *spread, zero before, becomes max_ij |out[i][j] - out[reader][j]|
// (null: not wanted).
bool gossip_step_applies(int32_t n);
bool gossip_joins(int32_t n, int chunks);
cudaError_t launch_gossip_step(const float *W, const float *partial, int chunks, const float *P, int32_t n, int32_t m, int32_t rounds,
                               float *out, int32_t reader, float *spread, cudaStream_t stream);
// `rounds` of them: P and scratch (n x m each) are both written, *result tells which holds the outcome.
cudaError_t launch_gossip_rounds(const float *W, float *P, int32_t n, int32_t m, int32_t rounds, float *scratch, float **result,
                                 cudaStream_t stream);
// spread[0] = max_ij |P[i*m + j] - P[reader*m + j]|
cudaError_t launch_consensus_spread(const float *P, int32_t n, int32_t m, int32_t reader, float *spread,
                                    cudaStream_t stream);

}  // namespace core
