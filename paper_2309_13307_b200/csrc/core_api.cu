// C ABI of the CORE library: argument checks, context, workspace and stream plumbing.
// Every entry point is declared, with its contract, in include/core.h.
#include "core.h"

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <new>
#include <utility>

#include "core_internal.h"
#include "core_sync.cuh"

using namespace core;

namespace core {

cudaError_t allow_shared(const void *kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    int device = 0;
    if (cudaError_t e = cudaGetDevice(&device)) return e;
    static std::mutex mutex;
    static std::map<std::pair<int, const void *>, size_t> granted;        // one entry per kernel and device
    std::lock_guard<std::mutex> lock(mutex);
    size_t &most = granted[{device, kernel}];
    if (bytes <= most) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) most = bytes;
    return e;
}

}  // namespace core

struct core_ctx {
    uint64_t seed;
    int64_t d;
    int32_t m;
    uint32_t t;
    int device;
    int sm_count;
    cudaStream_t stream;
    RoundKeys keys;
    void *ws;            // device workspace, grown on demand
    size_t ws_bytes;
    float *pbar;         // m floats, for callers that do not keep the message (gd step)
    int last_cuda;
    // host-streaming state (core_round_host), created on first use
    cudaStream_t copy_stream, work_stream;
    cudaEvent_t in_ready[2], in_free[2], out_ready[2], out_free[2];
    bool host_ready;
    void *slab;          // 2 input slabs + 2 output slabs
    size_t slab_bytes;
};

struct core_ls {
    const float *A;
    const float *b;
    int32_t n, rows;
    int64_t d;
    int device;
    LsPass step_pass;    // one pass over A, the machines' gradients added up (for the steps)
    LsPass machine_pass; // one pass over A, one gradient per machine
    LsPlan plan;         // two passes over A, where rows are too long for one (step_pass.units == 0)
    float *res;          // n*rows, two passes only
    float *part;         // partial gradients
    float *G;            // n*d
    float *y;            // d: look-ahead point of the accelerated step / trial point of the guarded step
    double *f_parts;     // loss at the trial point, one sum per unit of step_pass (or one in all)
    double *loss;        // loss on its way to the host
    int *accepted;       // 1 if the last guarded step took the trial point
    float *step;         // step chosen on the device (Option I of Algorithm 3), then its statistic p
};

namespace {

size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

int cuda_fail(core_ctx *ctx, cudaError_t e) {
    if (ctx) ctx->last_cuda = (int)e;
    return e == cudaErrorMemoryAllocation ? CORE_ENOMEM : CORE_ECUDA;
}

#define CORE_CUDA(ctx, expr)                                  \
    do {                                                      \
        cudaError_t e__ = (expr);                             \
        if (e__ != cudaSuccess) return cuda_fail((ctx), e__); \
    } while (0)

// Every device allocation of the library goes through here, so that tests can make the next ones fail
// on the host (core_debug_fail_allocations) and see the out-of-memory paths without exhausting a GPU.
std::atomic<int> g_fail_allocations{0};

cudaError_t core_malloc(void **out, size_t bytes) {
    int left = g_fail_allocations.load();
    while (left > 0) {
        if (g_fail_allocations.compare_exchange_weak(left, left - 1)) {
            *out = nullptr;
            return cudaErrorMemoryAllocation;
        }
    }
    return cudaMalloc(out, bytes);
}

bool on_device(int device) {
    int cur = -1;
    return cudaGetDevice(&cur) == cudaSuccess && cur == device;
}

int ensure_workspace(core_ctx *ctx, size_t bytes) {
    if (bytes <= ctx->ws_bytes) return CORE_OK;
    if (ctx->ws) {
        cudaError_t e = cudaFree(ctx->ws);   // waits for work that may still use it
        ctx->ws = nullptr;
        ctx->ws_bytes = 0;
        if (e != cudaSuccess) return cuda_fail(ctx, e);
    }
    bytes = round_up(bytes, (size_t)1 << 20);
    cudaError_t e = core_malloc(&ctx->ws, bytes);
    if (e != cudaSuccess) {
        ctx->ws = nullptr;
        cudaGetLastError();
        ctx->last_cuda = (int)e;
        return CORE_ENOMEM;
    }
    ctx->ws_bytes = bytes;
    return CORE_OK;
}

bool valid_dtype(int dtype) { return dtype == CORE_F32 || dtype == CORE_BF16; }
size_t elem_size(int dtype) { return dtype == CORE_BF16 ? 2 : 4; }

// One machine's message comes from the single-row kernel (unless a test asks for one of the others).
bool single_row(int32_t n) { return n == 1 && !project_kernel_forced(); }

// Rounds of several machines whose messages nobody asks for: the mean message is linear in the gradients, so
// the projection can add them up first and make one message instead of n.  That saves the n - 1 further
// multiply-adds per Gaussian (a quarter of the projection at n = 8, a third at n = 32).  Below 2^25 Gaussians
// (about 28 us of generating) the messages are formed one by one, so that a short round keeps giving the bits
// of core_project + core_aggregate.
constexpr int64_t kCombineFirst = (int64_t)1 << 25;
bool combine_first(const core_ctx *ctx, int32_t n) {
    return n > 1 && !project_kernel_forced() && ctx->d >= (kCombineFirst + ctx->m - 1) / ctx->m;
}

// A short vector's round of n machines goes through one kernel, and so does the projection of one (unless a test asks for one of the others).
ShortPlan short_plan(const core_ctx *ctx, int32_t n) {
    return project_kernel_forced() || short_kernels_off() ? ShortPlan{} : make_short_plan(n, 1, ctx->m, ctx->d, ctx->sm_count);
}

size_t row_partial_bytes(const core_ctx *ctx, int64_t d) {
    return round_up((size_t)row_plan_columns(ctx->m, d, ctx->sm_count) * ctx->m * sizeof(float), 256);
}

// Bytes of partial sums the projection of n machines needs (largest group of a pass).
size_t partial_bytes(const core_ctx *ctx, int32_t n, int64_t d, int dtype) {
    size_t need = row_partial_bytes(ctx, d);
    for (int32_t i0 = 0, ng = 0; i0 < n; i0 += ng) {
        ng = project_group(n - i0, ctx->m);
        const ProjectPlan plan = make_project_plan(ng, ctx->m, d, dtype, ctx->sm_count);
        const size_t b = (size_t)plan.grid_x * ng * ctx->m * sizeof(float);
        if (b > need) need = b;
    }
    return round_up(need, 256);
}

// message (m floats) = <scale * sum of `rows` rows, xi_j> over coordinates [0, d), added to what is there if asked.
int project_row_into(core_ctx *ctx, const void *G, int dtype, int32_t rows, int64_t ldg, float scale, int64_t d,
                     uint64_t q_base, float *partial, float *message, bool accumulate, cudaStream_t stream) {
    const RowPlan plan = make_row_plan(G, dtype, rows, ldg, ctx->m, d, ctx->sm_count);
    CORE_CUDA(ctx, launch_project_row(plan, ctx->keys, ctx->t, G, dtype, rows, ldg, scale, d, ctx->m, q_base, partial, stream));
    CORE_CUDA(ctx, launch_finish_project(partial, plan.grid_x, 1, ctx->m, message, accumulate, stream));
    return CORE_OK;
}

// Projects rows [0, n) of a matrix whose coordinate 0 is global block q_base; the partial
// sums go through `partial`; P (n*m) receives (or accumulates) the result.
int project_into(core_ctx *ctx, const void *G, int dtype, int32_t n, int64_t ldg, int64_t d, uint64_t q_base,
                 float *partial, float *P, bool accumulate, cudaStream_t stream) {
    if (single_row(n)) return project_row_into(ctx, G, dtype, 1, ldg, 1.0f, d, q_base, partial, P, accumulate, stream);
    for (int32_t i0 = 0, ng = 0; i0 < n; i0 += ng) {
        ng = project_group(n - i0, ctx->m);
        const ProjectPlan plan = make_project_plan(ng, ctx->m, d, dtype, ctx->sm_count);
        const char *rows = static_cast<const char *>(G) + (size_t)i0 * (size_t)ldg * elem_size(dtype);
        CORE_CUDA(ctx, launch_project(plan, ctx->keys, ctx->t, rows, dtype, ng, ldg, d, ctx->m, q_base, partial,
                                      stream));
        CORE_CUDA(ctx, launch_finish_project(partial, plan.grid_x, ng, ctx->m, P + (size_t)i0 * ctx->m, accumulate,
                                             stream));
    }
    return CORE_OK;
}

// The messages of n machines' whole vectors.
int project_all(core_ctx *ctx, const void *G, int dtype, int32_t n, int64_t ldg, float *partial, float *P) {
    const ShortPlan plan = n == 1 ? short_plan(ctx, 1) : ShortPlan{};
    if (plan.ctas == 0) return project_into(ctx, G, dtype, n, ldg, ctx->d, 0, partial, P, false, ctx->stream);
    CORE_CUDA(ctx, launch_short_round(plan, ctx->keys, ctx->t, G, dtype, 1, n, ldg, 1.0f, ctx->d, ctx->m, P, nullptr, nullptr, nullptr, ctx->stream));
    return CORE_OK;
}

// The estimate of the whole vector, or the update made from it.
int reconstruct_all(core_ctx *ctx, float *pbar, float *out, const ReconstructEpilogue *epilogue, const MessageParts *parts = nullptr) {
    const ShortPlan plan = short_kernels_off() ? ShortPlan{} : make_short_plan(1, 1, ctx->m, ctx->d, ctx->sm_count);
    if (plan.ctas > 0)
        CORE_CUDA(ctx, launch_short_reconstruct(plan, ctx->keys, ctx->t, pbar, ctx->d, ctx->m, out, ctx->sm_count, epilogue, parts, ctx->stream));
    else
        CORE_CUDA(ctx, launch_reconstruct(ctx->keys, ctx->t, pbar, ctx->m, 0, ctx->d, out, ctx->sm_count, ctx->stream, epilogue, parts));
    return CORE_OK;
}

int check_ctx(const core_ctx *ctx) {
    if (!ctx) return CORE_EINVAL;
    if (!on_device(ctx->device)) return CORE_EINVAL;
    return CORE_OK;
}

}  // namespace

extern "C" {

int core_init(core_ctx **out, uint64_t seed, int64_t d, int32_t m) {
    if (!out) return CORE_EINVAL;
    *out = nullptr;
    if (d < 1 || m < 1) return CORE_EINVAL;
    core_ctx *ctx = new (std::nothrow) core_ctx();
    if (!ctx) return CORE_ENOMEM;
    ctx->seed = seed;
    ctx->d = d;
    ctx->m = m;
    ctx->t = 0;
    ctx->stream = nullptr;
    ctx->keys = expand_keys(seed);
    ctx->ws = nullptr;
    ctx->ws_bytes = 0;
    ctx->pbar = nullptr;
    ctx->last_cuda = 0;
    ctx->host_ready = false;
    ctx->slab = nullptr;
    ctx->slab_bytes = 0;
    cudaError_t e = cudaGetDevice(&ctx->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, ctx->device);
    if (e == cudaSuccess) e = core_malloc(reinterpret_cast<void **>(&ctx->pbar), (size_t)m * sizeof(float));
    if (e != cudaSuccess) {
        cudaGetLastError();
        const int rc = e == cudaErrorMemoryAllocation ? CORE_ENOMEM : CORE_ECUDA;
        delete ctx;
        return rc;
    }
    *out = ctx;
    return CORE_OK;
}

int core_destroy(core_ctx *ctx) {
    if (!ctx) return CORE_EINVAL;
    int rc = CORE_OK;
    if (ctx->ws && cudaFree(ctx->ws) != cudaSuccess) rc = CORE_ECUDA;
    if (ctx->pbar && cudaFree(ctx->pbar) != cudaSuccess) rc = CORE_ECUDA;
    if (ctx->slab && cudaFree(ctx->slab) != cudaSuccess) rc = CORE_ECUDA;
    if (ctx->host_ready) {
        cudaStreamDestroy(ctx->copy_stream);
        cudaStreamDestroy(ctx->work_stream);
        for (int s = 0; s < 2; ++s) {
            cudaEventDestroy(ctx->in_ready[s]);
            cudaEventDestroy(ctx->in_free[s]);
            cudaEventDestroy(ctx->out_ready[s]);
            cudaEventDestroy(ctx->out_free[s]);
        }
    }
    delete ctx;
    return rc;
}

int core_set_stream(core_ctx *ctx, void *cuda_stream) {
    if (!ctx) return CORE_EINVAL;
    ctx->stream = static_cast<cudaStream_t>(cuda_stream);
    return CORE_OK;
}

int core_set_round(core_ctx *ctx, uint32_t t) {
    if (!ctx) return CORE_EINVAL;
    ctx->t = t;
    return CORE_OK;
}

uint32_t core_get_round(const core_ctx *ctx) { return ctx ? ctx->t : 0u; }

size_t core_workspace_bytes(const core_ctx *ctx) {
    return ctx ? ctx->ws_bytes + ctx->slab_bytes + (size_t)ctx->m * sizeof(float) : 0;
}

const char *core_strerror(int code) {
    switch (code) {
        case CORE_OK: return "ok";
        case CORE_EINVAL: return "invalid argument";
        case CORE_ENOMEM: return "out of device memory";
        case CORE_ECUDA: return "CUDA runtime error";
        case CORE_ELIMIT: return "size exceeds the fixed capacity of this entry point";
        default: return "unknown error";
    }
}

int core_last_cuda_error(const core_ctx *ctx) { return ctx ? ctx->last_cuda : 0; }

int core_device_status(int32_t *status_out) {
    if (!status_out) return CORE_EINVAL;
    int status = 0;
    if (project_tc_take_status(&status) != cudaSuccess) {
        cudaGetLastError();
        return CORE_ECUDA;
    }
    int pass = 0;
    if (ls_pass_take_status(&pass) != cudaSuccess) {
        cudaGetLastError();
        return CORE_ECUDA;
    }
    *status_out = status > pass ? status : pass;
    return CORE_OK;
}

int core_project(core_ctx *ctx, const void *G_dev, int dtype, int32_t n, int64_t ldg, float *P_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!G_dev || !P_dev || n < 1 || ldg < ctx->d || !valid_dtype(dtype)) return CORE_EINVAL;
    if (int rc = ensure_workspace(ctx, partial_bytes(ctx, n, ctx->d, dtype))) return rc;
    return project_all(ctx, G_dev, dtype, n, ldg, static_cast<float *>(ctx->ws), P_dev);
}

int core_reserve_workspace(core_ctx *ctx, int32_t n, int dtype) {
    if (int rc = check_ctx(ctx)) return rc;
    if (n < 1 || !valid_dtype(dtype)) return CORE_EINVAL;
    // what core_round needs (partial sums + the messages); core_project needs the first part only
    const size_t pb = partial_bytes(ctx, n, ctx->d, dtype);
    const size_t Pb = round_up((size_t)n * ctx->m * sizeof(float), 256);
    return ensure_workspace(ctx, pb + Pb);
}

int core_aggregate(core_ctx *ctx, const float *P_dev, int32_t n, float *pbar_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!P_dev || !pbar_dev || n < 1) return CORE_EINVAL;
    CORE_CUDA(ctx, launch_aggregate(P_dev, n, ctx->m, pbar_dev, ctx->stream));
    return CORE_OK;
}

int core_reconstruct(core_ctx *ctx, const float *pbar_dev, float *gtilde_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!pbar_dev || !gtilde_dev) return CORE_EINVAL;
    return reconstruct_all(ctx, const_cast<float *>(pbar_dev), gtilde_dev, nullptr);
}

// A step chosen on the device from the combined messages, between aggregation and reconstruction
// (Option I of Algorithm 3): h_dev receives the step, p_dev (may be null) the statistic.
struct StepRule {
    double r1, H, c;
    float *p_dev;
    float *h_dev;
};

static int apply_step_rule(core_ctx *ctx, const StepRule *rule, const float *pbar_dev) {
    if (!rule) return CORE_OK;
    CORE_CUDA(ctx, launch_option1_step(pbar_dev, ctx->m, ctx->d, rule->r1, rule->H, rule->c, rule->p_dev, rule->h_dev,
                                       ctx->stream));
    return CORE_OK;
}

// The round of one combined row (see launch_project_row): message, step rule, reconstruction, then t <- t + 1.  A short
// round leaves it to the reconstruction to finish the message.
static int finish_round(core_ctx *ctx, const void *G, int dtype, int32_t rows, int64_t ldg, float scale, float *partial,
                        float *pbar_dev, float *out, const ReconstructEpilogue *epilogue, const StepRule *rule) {
    const RowPlan plan = make_row_plan(G, dtype, rows, ldg, ctx->m, ctx->d, ctx->sm_count);
    CORE_CUDA(ctx, launch_project_row(plan, ctx->keys, ctx->t, G, dtype, rows, ldg, scale, ctx->d, ctx->m, 0, partial, ctx->stream));
    if (!rule && reconstruct_joins(plan.grid_x, 1, ctx->m, ctx->d, ctx->sm_count)) {
        const MessageParts parts{partial, plan.grid_x, 1};
        if (int rc = reconstruct_all(ctx, pbar_dev, out, epilogue, &parts)) return rc;
    } else {
        CORE_CUDA(ctx, launch_finish_project(partial, plan.grid_x, 1, ctx->m, pbar_dev, false, ctx->stream));
        if (int rc = apply_step_rule(ctx, rule, pbar_dev)) return rc;
        if (int rc = reconstruct_all(ctx, pbar_dev, out, epilogue)) return rc;
    }
    ctx->t += 1;
    return CORE_OK;
}

// project -> aggregate -> reconstruct with the current t, then t <- t + 1.  With an epilogue the
// reconstruction writes the optimiser update into `out` instead of the estimate.
static int round_with_epilogue(core_ctx *ctx, const void *G_dev, int dtype, int32_t n, int64_t ldg, float *pbar_dev,
                               float *out, const ReconstructEpilogue *epilogue, const StepRule *rule = nullptr) {
    const size_t pb = partial_bytes(ctx, n, ctx->d, dtype);
    const size_t Pb = round_up((size_t)n * ctx->m * sizeof(float), 256);
    if (int rc = ensure_workspace(ctx, pb + Pb)) return rc;
    float *partial = static_cast<float *>(ctx->ws);
    float *P = reinterpret_cast<float *>(static_cast<char *>(ctx->ws) + pb);
    const ShortPlan in_one = short_plan(ctx, n);
    if (in_one.ctas > 0 && !rule) {
        CORE_CUDA(ctx, launch_short_round(in_one, ctx->keys, ctx->t, G_dev, dtype, 1, n, ldg, 1.0f, ctx->d, ctx->m, nullptr, pbar_dev, out, epilogue,
                                          ctx->stream));
        ctx->t += 1;
        return CORE_OK;
    }
    if (single_row(n) || combine_first(ctx, n))
        return finish_round(ctx, G_dev, dtype, n, ldg, 1.0f / (float)n, partial, pbar_dev, out, epilogue, rule);
    if (project_group(n, ctx->m) == n) {
        // one group of machines: the per-machine messages are not kept, so they are never written
        const ProjectPlan plan = make_project_plan(n, ctx->m, ctx->d, dtype, ctx->sm_count);
        CORE_CUDA(ctx, launch_project(plan, ctx->keys, ctx->t, G_dev, dtype, n, ldg, ctx->d, ctx->m, 0, partial,
                                      ctx->stream));
        if (!rule && reconstruct_joins(plan.grid_x, n, ctx->m, ctx->d, ctx->sm_count)) {
            const MessageParts parts{partial, plan.grid_x, n};
            if (int rc = reconstruct_all(ctx, pbar_dev, out, epilogue, &parts)) return rc;
            ctx->t += 1;
            return CORE_OK;
        }
        CORE_CUDA(ctx, launch_finish_aggregate(partial, plan.grid_x, n, ctx->m, pbar_dev, ctx->stream));
    } else {
        if (int rc = project_all(ctx, G_dev, dtype, n, ldg, partial, P)) return rc;
        CORE_CUDA(ctx, launch_aggregate(P, n, ctx->m, pbar_dev, ctx->stream));
    }
    if (int rc = apply_step_rule(ctx, rule, pbar_dev)) return rc;
    if (int rc = reconstruct_all(ctx, pbar_dev, out, epilogue)) return rc;
    ctx->t += 1;
    return CORE_OK;
}

int core_round(core_ctx *ctx, const void *G_dev, int dtype, int32_t n, int64_t ldg, float *pbar_dev,
               float *gtilde_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!G_dev || !pbar_dev || !gtilde_dev || n < 1 || ldg < ctx->d || !valid_dtype(dtype)) return CORE_EINVAL;
    return round_with_epilogue(ctx, G_dev, dtype, n, ldg, pbar_dev, gtilde_dev, nullptr);
}

static int round_host_body(core_ctx *ctx, const void *G_host, int dtype, int32_t n, int64_t ldg, float *pbar_host,
                           float *gtilde_host);

int core_round_host(core_ctx *ctx, const void *G_host, int dtype, int32_t n, int64_t ldg, float *pbar_host,
                    float *gtilde_host) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!G_host || !pbar_host || !gtilde_host || n < 1 || ldg < ctx->d || !valid_dtype(dtype)) return CORE_EINVAL;
    const int rc = round_host_body(ctx, G_host, dtype, n, ldg, pbar_host, gtilde_host);
    if (rc != CORE_OK && ctx->host_ready) {
        // copies enqueued before the failure may still be reading G_host or writing the outputs: the
        // caller gets its buffers back only once both streams have drained (a second error is ignored)
        const int first = ctx->last_cuda;
        cudaStreamSynchronize(ctx->work_stream);
        cudaStreamSynchronize(ctx->copy_stream);
        cudaGetLastError();
        ctx->last_cuda = first;
    }
    return rc;
}

// How a vector of a host round is cut into slabs: growing from `least` with what is behind them, shrinking to `least` with
// what is ahead, `most` at most, multiples of 4096 but for the end of the vector; from `whole_from` on whole multiples of `whole`.
struct SlabRule {
    int64_t least, most, whole_from, whole;
};
static int64_t next_slab(int64_t k0, int64_t d, const SlabRule &r) {
    const int64_t left = d - k0;
    int64_t len = std::min(r.most, std::min(k0 + r.least, std::max(left / 2, r.least)));
    len = std::max<int64_t>(len / 4096 * 4096, 4096);
    if (len >= r.whole_from) len = len / r.whole * r.whole;
    return left - len < r.least / 2 ? (left <= r.most ? left : len) : len;
}
static int64_t slab_limit(int64_t d, int64_t bytes, size_t per_coordinate) {
    const int64_t whole = (d + 4095) / 4096 * 4096, slab = bytes / (int64_t)per_coordinate / 4096 * 4096;
    return slab < 4096 ? 4096 : slab > whole ? whole : slab;
}
// Slabs of at most 64 MiB of input over all machines and 16 MiB of output.  The first and the last ones are shorter: what is
// not overlapped is the projection of the last slab and the reconstruction of the first one (and, where the kernels
// are the slower side, the first copy in and the last out).
static SlabRule input_slabs(int64_t d, int32_t n, size_t es) {
    const int64_t most = slab_limit(d, (int64_t)64 << 20, es * (size_t)n);
    // at least 256 KB per machine and copy
    return {std::min(most, slab_limit(d, std::max((int64_t)4 << 20, (int64_t)n << 18), es * (size_t)n)), most, INT64_MAX, 1};
}
// Every slab is one launch of the reconstruction.  Long slabs are whole multiples of 48 units of 32 blocks per SM, at most four
// of them on 148 SMs: with the table of angles every SM has the same number of units then (six per warp in the longest slabs), and
// 48 units are also one wave of the kernel for few or very many vectors.  (Longest slabs of eight multiples: longer steps up to
// them where the copies are the slower side: n = 1, d = 3e7, m = 64: 4.80 -> 4.90 ms.)
static SlabRule output_slabs(int64_t d, int sm_count) {
    const int64_t most = slab_limit(d, (int64_t)16 << 20, sizeof(float));
    return {std::min(most, slab_limit(d, (int64_t)1 << 20, sizeof(float))), most,
            (int64_t)sm_count << 14, 3 * ((int64_t)sm_count << 11)};
}

static int round_host_body(core_ctx *ctx, const void *G_host, int dtype, int32_t n, int64_t ldg, float *pbar_host,
                           float *gtilde_host) {
    if (!ctx->host_ready) {
        // all or nothing: a half-made set of streams and events is torn down again
        cudaError_t e = cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
        e = cudaStreamCreateWithFlags(&ctx->work_stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            cudaStreamDestroy(ctx->copy_stream);
            return cuda_fail(ctx, e);
        }
        cudaEvent_t *events[8] = {&ctx->in_ready[0], &ctx->in_ready[1], &ctx->in_free[0], &ctx->in_free[1],
                                  &ctx->out_ready[0], &ctx->out_ready[1], &ctx->out_free[0], &ctx->out_free[1]};
        int made = 0;
        for (; made < 8 && e == cudaSuccess; ++made) e = cudaEventCreateWithFlags(events[made], cudaEventDisableTiming);
        if (e != cudaSuccess) {
            for (int k = 0; k + 1 < made; ++k) cudaEventDestroy(*events[k]);
            cudaStreamDestroy(ctx->copy_stream);
            cudaStreamDestroy(ctx->work_stream);
            return cuda_fail(ctx, e);
        }
        ctx->host_ready = true;
    }
    const size_t es = elem_size(dtype);
    const int64_t d = ctx->d;
    const SlabRule in = input_slabs(d, n, es), out = output_slabs(d, ctx->sm_count);
    // the longest ones that occur, and the partial sums any of them needs
    int64_t in_len = 0, out_len = 0;
    size_t pb = 0;
    for (int64_t k0 = 0, len = 0; k0 < d; k0 += len) {
        len = next_slab(k0, d, in);
        if (len > in_len) in_len = len;
        pb = std::max(pb, row_partial_bytes(ctx, len));
    }
    for (int64_t k0 = 0, len = 0; k0 < d; k0 += len) {
        len = next_slab(k0, d, out);
        if (len > out_len) out_len = len;
    }
    in_len = (in_len + 7) / 8 * 8;                      // rows of a slab start on 16 bytes
    const size_t in_bytes = round_up((size_t)n * (size_t)in_len * es, 256);
    const size_t out_bytes = round_up((size_t)out_len * sizeof(float), 256);
    const size_t need_slab = 2 * in_bytes + 2 * out_bytes;
    if (need_slab > ctx->slab_bytes) {
        if (ctx->slab) {
            cudaFree(ctx->slab);
            ctx->slab = nullptr;
            ctx->slab_bytes = 0;
        }
        cudaError_t e = core_malloc(&ctx->slab, need_slab);
        if (e != cudaSuccess) {
            cudaGetLastError();
            ctx->last_cuda = (int)e;
            return CORE_ENOMEM;
        }
        ctx->slab_bytes = need_slab;
    }
    const size_t mb = round_up((size_t)ctx->m * sizeof(float), 256);
    if (int rc = ensure_workspace(ctx, pb + mb)) return rc;
    char *in_buf[2] = {static_cast<char *>(ctx->slab), static_cast<char *>(ctx->slab) + in_bytes};
    float *out_buf[2] = {reinterpret_cast<float *>(static_cast<char *>(ctx->slab) + 2 * in_bytes),
                         reinterpret_cast<float *>(static_cast<char *>(ctx->slab) + 2 * in_bytes + out_bytes)};
    float *partial = static_cast<float *>(ctx->ws);
    float *pbar = reinterpret_cast<float *>(static_cast<char *>(ctx->ws) + pb);

    CORE_CUDA(ctx, cudaStreamSynchronize(ctx->stream));   // earlier work of the caller on this context

    // projection: slab s is copied while slab s-1 is projected; the mean message grows slab by slab (the gradients of a
    // slab are added while they are staged)
    int64_t len = 0;
    int s = 0;
    for (int64_t k0 = 0; k0 < d; k0 += len, ++s) {
        const int b = s & 1;
        len = next_slab(k0, d, in);
        if (s >= 2) CORE_CUDA(ctx, cudaStreamWaitEvent(ctx->copy_stream, ctx->in_free[b], 0));
        const char *const from = static_cast<const char *>(G_host) + (size_t)k0 * es;
        if ((size_t)ldg * es <= (size_t)INT32_MAX)          // one copy for all rows, where the stride is a legal pitch
            CORE_CUDA(ctx, cudaMemcpy2DAsync(in_buf[b], (size_t)in_len * es, from, (size_t)ldg * es, (size_t)len * es, (size_t)n,
                                             cudaMemcpyHostToDevice, ctx->copy_stream));
        else
            for (int32_t i = 0; i < n; ++i)
                CORE_CUDA(ctx, cudaMemcpyAsync(in_buf[b] + (size_t)i * (size_t)in_len * es, from + (size_t)i * (size_t)ldg * es,
                                               (size_t)len * es, cudaMemcpyHostToDevice, ctx->copy_stream));
        CORE_CUDA(ctx, cudaEventRecord(ctx->in_ready[b], ctx->copy_stream));
        CORE_CUDA(ctx, cudaStreamWaitEvent(ctx->work_stream, ctx->in_ready[b], 0));
        if (int rc = project_row_into(ctx, in_buf[b], dtype, n, in_len, 1.0f / (float)n, len, (uint64_t)k0 >> 2, partial, pbar,
                                      s > 0, ctx->work_stream))
            return rc;
        CORE_CUDA(ctx, cudaEventRecord(ctx->in_free[b], ctx->work_stream));
    }
    // the last slab's event also tells that the message is complete
    CORE_CUDA(ctx, cudaStreamWaitEvent(ctx->copy_stream, ctx->in_free[(s - 1) & 1], 0));
    CORE_CUDA(ctx, cudaMemcpyAsync(pbar_host, pbar, (size_t)ctx->m * sizeof(float), cudaMemcpyDeviceToHost, ctx->copy_stream));
    // reconstruction: slab s is copied back while slab s+1 is generated
    s = 0;
    for (int64_t k0 = 0; k0 < d; k0 += len, ++s) {
        const int b = s & 1;
        len = next_slab(k0, d, out);
        if (s >= 2) CORE_CUDA(ctx, cudaStreamWaitEvent(ctx->work_stream, ctx->out_free[b], 0));
        CORE_CUDA(ctx, launch_reconstruct(ctx->keys, ctx->t, pbar, ctx->m, k0, k0 + len, out_buf[b], ctx->sm_count,
                                          ctx->work_stream));
        CORE_CUDA(ctx, cudaEventRecord(ctx->out_ready[b], ctx->work_stream));
        CORE_CUDA(ctx, cudaStreamWaitEvent(ctx->copy_stream, ctx->out_ready[b], 0));
        CORE_CUDA(ctx, cudaMemcpyAsync(gtilde_host + k0, out_buf[b], (size_t)len * sizeof(float),
                                       cudaMemcpyDeviceToHost, ctx->copy_stream));
        CORE_CUDA(ctx, cudaEventRecord(ctx->out_free[b], ctx->copy_stream));
    }
    CORE_CUDA(ctx, cudaStreamSynchronize(ctx->work_stream));
    CORE_CUDA(ctx, cudaStreamSynchronize(ctx->copy_stream));
    ctx->t += 1;
    return CORE_OK;
}

/* ---- least squares ---------------------------------------------------------- */

int core_ls_create(core_ls **out, const float *A_dev, const float *b_dev, int32_t n, int32_t rows, int64_t d) {
    if (!out) return CORE_EINVAL;
    *out = nullptr;
    if (!A_dev || !b_dev || n < 1 || rows < 1 || d < 1) return CORE_EINVAL;
    core_ls *ls = new (std::nothrow) core_ls();
    if (!ls) return CORE_ENOMEM;
    ls->A = A_dev;
    ls->b = b_dev;
    ls->n = n;
    ls->rows = rows;
    ls->d = d;
    int sm = 0;
    cudaError_t e = cudaGetDevice(&ls->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, ls->device);
    if (e != cudaSuccess) {
        delete ls;
        return CORE_ECUDA;
    }
    ls->step_pass = make_ls_pass(n, rows, d, false, sm);
    ls->machine_pass = make_ls_pass(n, rows, d, true, sm);
    if (ls->machine_pass.units == 0) ls->step_pass = LsPass{};
    const bool one_pass = ls->step_pass.units > 0;
    size_t part = 0;
    if (one_pass) {
        const size_t together = ls_pass_partials(ls->step_pass), apart = ls_pass_partials(ls->machine_pass);
        part = std::max(together, apart);
    } else {
        ls->plan = make_ls_plan(n, rows, d, sm);
        part = (size_t)n * ls->plan.splits * (size_t)d;
    }
    const size_t res_b = one_pass ? 256 : round_up((size_t)n * rows * sizeof(float), 256);
    const size_t part_b = round_up(part * sizeof(float), 256);
    const size_t G_b = round_up((size_t)n * (size_t)d * sizeof(float), 256);
    const size_t gt_b = round_up((size_t)d * sizeof(float), 256);
    const size_t f_b = round_up((size_t)(one_pass ? ls->step_pass.units : 1) * sizeof(double), 256);
    const size_t scalars_b = 256;                          // loss, acceptance flag, step and statistic
    char *base = nullptr;
    e = core_malloc(reinterpret_cast<void **>(&base), res_b + part_b + G_b + gt_b + f_b + scalars_b);
    if (e != cudaSuccess) {
        cudaGetLastError();
        delete ls;
        return CORE_ENOMEM;
    }
    ls->res = reinterpret_cast<float *>(base);
    ls->part = reinterpret_cast<float *>(base + res_b);
    ls->G = reinterpret_cast<float *>(base + res_b + part_b);
    ls->y = reinterpret_cast<float *>(base + res_b + part_b + G_b);
    ls->f_parts = reinterpret_cast<double *>(base + res_b + part_b + G_b + gt_b);
    char *const scalars = base + res_b + part_b + G_b + gt_b + f_b;
    ls->loss = reinterpret_cast<double *>(scalars);
    ls->accepted = reinterpret_cast<int *>(scalars + 16);
    ls->step = reinterpret_cast<float *>(scalars + 32);
    *out = ls;
    return CORE_OK;
}

int core_ls_destroy(core_ls *ls) {
    if (!ls) return CORE_EINVAL;
    const int rc = cudaFree(ls->res) == cudaSuccess ? CORE_OK : CORE_ECUDA;   // res is the base of the block
    delete ls;
    return rc;
}

static int ls_gradients_into(core_ctx *ctx, core_ls *ls, const float *x_dev, float *G, float *clear = nullptr) {
    if (ls->machine_pass.units > 0) {
        CORE_CUDA(ctx, launch_ls_pass_gradients(ls->machine_pass, ls->A, ls->b, LsPoint{x_dev}, ls->d, ls->part, ctx->stream));
        CORE_CUDA(ctx, launch_ls_pass_reduce(ls->machine_pass, ls->part, ls->d, 1.0f / (float)ls->rows, G, clear, ctx->stream));
        return CORE_OK;
    }
    CORE_CUDA(ctx, launch_ls_residual(ls->A, ls->b, x_dev, ls->n, ls->rows, ls->d, ls->res, ctx->stream));
    CORE_CUDA(ctx, launch_ls_at_r(ls->plan, ls->A, ls->res, ls->n, ls->rows, ls->d, ls->part, ctx->stream));
    CORE_CUDA(ctx, launch_ls_reduce(ls->plan, ls->part, ls->n, ls->rows, ls->d, G, clear, ctx->stream));
    return CORE_OK;
}

static double ls_loss_scale(const core_ls *ls) { return 1.0 / (2.0 * (double)ls->rows * (double)ls->n); }

// The objective at x as unscaled sums in ls->f_parts; returns how many through *parts.
static int ls_loss_parts(core_ctx *ctx, core_ls *ls, const float *x, bool reverse, int64_t *parts) {
    if (ls->step_pass.units > 0) {
        CORE_CUDA(ctx, launch_ls_pass_loss(ls->step_pass, ls->A, ls->b, LsPoint{x}, ls->d, reverse, ls->f_parts, ctx->stream));
        *parts = ls->step_pass.units;
        return CORE_OK;
    }
    CORE_CUDA(ctx, launch_ls_residual(ls->A, ls->b, x, ls->n, ls->rows, ls->d, ls->res, ctx->stream));
    CORE_CUDA(ctx, launch_ls_loss(ls->res, ls->n, ls->rows, ls->f_parts, ctx->stream));
    *parts = 1;
    return CORE_OK;
}

static int ls_loss_into(core_ctx *ctx, core_ls *ls, const float *x, double *loss) {
    int64_t parts = 0;
    if (int rc = ls_loss_parts(ctx, ls, x, false, &parts)) return rc;
    CORE_CUDA(ctx, launch_ls_loss_sum(ls->f_parts, parts, ls_loss_scale(ls), loss, ctx->stream));
    return CORE_OK;
}

// The round of one combined gradient, scale times the sum of `count` rows, of a context's whole vector.
static int combined_round(core_ctx *ctx, const float *rows, int32_t count, int64_t ld, float scale, float *pbar, float *out,
                          const ReconstructEpilogue *epilogue, const StepRule *rule) {
    const ShortPlan plan = short_kernels_off() ? ShortPlan{} : make_short_plan(1, count, ctx->m, ctx->d, ctx->sm_count);
    if (plan.ctas > 0 && !rule) {
        CORE_CUDA(ctx, launch_short_round(plan, ctx->keys, ctx->t, rows, CORE_F32, count, 1, ld, scale, ctx->d, ctx->m, nullptr, pbar, out, epilogue,
                                          ctx->stream));
        ctx->t += 1;
        return CORE_OK;
    }
    if (int rc = ensure_workspace(ctx, row_partial_bytes(ctx, ctx->d))) return rc;
    return finish_round(ctx, rows, CORE_F32, count, ld, scale, static_cast<float *>(ctx->ws), pbar, out, epilogue, rule);
}

// The round of a step at the point `at`: only the mean message is wanted, so the gradient is one row.  The
// projection adds the units' partial gradients while it stages its tiles; the machine gradients are never written.
static int ls_round(core_ctx *ctx, core_ls *ls, const LsPoint &at, float *out, const ReconstructEpilogue *epilogue,
                    const StepRule *rule = nullptr) {
    const float *rows = ls->part;
    int32_t count = (int32_t)ls->step_pass.units;
    int64_t ld = ls->step_pass.ldp;
    float scale = 1.0f / ((float)ls->rows * (float)ls->n);
    if (ls->step_pass.units > 0) {
        CORE_CUDA(ctx, launch_ls_pass_gradients(ls->step_pass, ls->A, ls->b, at, ls->d, ls->part, ctx->stream));
    } else {
        const float *x = at.x;
        if (at.x_prev) {
            CORE_CUDA(ctx, launch_lookahead(at.x, at.x_prev, at.gamma, ls->d, ls->y, ctx->stream));
            x = ls->y;
        }
        if (int rc = ls_gradients_into(ctx, ls, x, ls->G)) return rc;
        rows = ls->G;
        count = ls->n;
        ld = ls->d;
        scale = 1.0f / (float)ls->n;
    }
    return combined_round(ctx, rows, count, ld, scale, ctx->pbar, out, epilogue, rule);
}

int core_ls_gradients(core_ctx *ctx, core_ls *ls, const float *x_dev, float *G_out_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !x_dev || !G_out_dev || ls->d != ctx->d || ls->device != ctx->device) return CORE_EINVAL;
    return ls_gradients_into(ctx, ls, x_dev, G_out_dev);
}

int core_gd_step(core_ctx *ctx, core_ls *ls, float h, float *x_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !x_dev || ls->d != ctx->d || ls->device != ctx->device) return CORE_EINVAL;
    // x <- x - h * gtilde inside the reconstruction: the estimate is never stored
    const ReconstructEpilogue update{x_dev, h, nullptr, nullptr};
    return ls_round(ctx, ls, LsPoint{x_dev}, x_dev, &update);
}

int core_agd_step(core_ctx *ctx, core_ls *ls, float h, float beta, float *x_dev, float *x_prev_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !x_dev || !x_prev_dev || x_dev == x_prev_dev || ls->d != ctx->d || ls->device != ctx->device)
        return CORE_EINVAL;
    // x_prev <- x and x <- y - h * gtilde(y), both inside the reconstruction, which forms y again from x and x_prev
    ReconstructEpilogue update{x_dev, h, x_dev, x_prev_dev};
    update.lookahead = true;
    update.gamma = 1.0f - beta;
    return ls_round(ctx, ls, LsPoint{x_dev, x_prev_dev, 1.0f - beta}, x_dev, &update);
}

int core_gd_step_guarded(core_ctx *ctx, core_ls *ls, float h, float *x_dev, double *f_dev, int32_t *accepted_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !x_dev || !f_dev || ls->d != ctx->d || ls->device != ctx->device) return CORE_EINVAL;
    // trial point y = x - h * gtilde, written by the reconstruction; x is left untouched
    const ReconstructEpilogue trial{x_dev, h, nullptr, nullptr};
    if (int rc = ls_round(ctx, ls, LsPoint{x_dev}, ls->y, &trial)) return rc;
    // the trial point's loss, from the rows the gradient pass read last (still in L2) to those it read first
    int64_t parts = 0;
    if (int rc = ls_loss_parts(ctx, ls, ls->y, true, &parts)) return rc;
    // decided on the device: no host synchronisation inside the step
    CORE_CUDA(ctx, launch_keep_better(ls->f_parts, parts, ls_loss_scale(ls), ls->y, ls->d, f_dev, x_dev, ls->accepted,
                                      accepted_dev, ctx->stream));
    return CORE_OK;
}

int core_gd_step_option1(core_ctx *ctx, core_ls *ls, double r1, double H, double c, float *x_dev, double *f_dev,
                         int32_t *accepted_dev, float *p_dev, float *h_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !x_dev || !f_dev || ls->d != ctx->d || ls->device != ctx->device || !(r1 > 0.0) || !(H > 0.0) ||
        !(c > 0.0))
        return CORE_EINVAL;
    // the step is formed on the device between aggregation and reconstruction; the reconstruction reads it
    // there and writes the trial point y = x - h * gtilde; x is left untouched until the comparison
    const StepRule rule{r1, H, c, ls->step + 1, ls->step};
    ReconstructEpilogue trial{x_dev, 0.f, nullptr, nullptr};
    trial.step_dev = ls->step;
    if (int rc = ls_round(ctx, ls, LsPoint{x_dev}, ls->y, &trial, &rule)) return rc;
    // the trial point's loss, from the rows the gradient pass read last (still in L2) to those it read first
    int64_t parts = 0;
    if (int rc = ls_loss_parts(ctx, ls, ls->y, true, &parts)) return rc;
    CORE_CUDA(ctx, launch_keep_better(ls->f_parts, parts, ls_loss_scale(ls), ls->y, ls->d, f_dev, x_dev, ls->accepted,
                                      accepted_dev, ctx->stream));
    if (h_dev)
        CORE_CUDA(ctx, cudaMemcpyAsync(h_dev, ls->step, sizeof(float), cudaMemcpyDeviceToDevice, ctx->stream));
    if (p_dev)
        CORE_CUDA(ctx, cudaMemcpyAsync(p_dev, ls->step + 1, sizeof(float), cudaMemcpyDeviceToDevice, ctx->stream));
    return CORE_OK;
}

int core_gossip_round(core_ctx *ctx, const float *W_dev, const float *P_in_dev, int32_t n, float *P_out_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!W_dev || !P_in_dev || !P_out_dev || P_in_dev == P_out_dev || n < 1) return CORE_EINVAL;
    CORE_CUDA(ctx, launch_gossip_round(W_dev, P_in_dev, n, ctx->m, P_out_dev, ctx->stream));
    return CORE_OK;
}

int core_decentralized_step(core_ctx *ctx, core_ls *ls, const float *W_dev, int32_t rounds, int32_t reader,
                            int as_printed, float h, float *x_dev, float *spread_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !W_dev || !x_dev || ls->d != ctx->d || ls->device != ctx->device || rounds < 0 || reader < 0 ||
        reader >= ls->n)
        return CORE_EINVAL;
    const int32_t n = ls->n;
    const size_t pb = partial_bytes(ctx, n, ctx->d, CORE_F32);
    const size_t Pb = round_up((size_t)n * ctx->m * sizeof(float), 256);
    if (int rc = ensure_workspace(ctx, pb + 2 * Pb)) return rc;
    float *partial = static_cast<float *>(ctx->ws);
    float *P = reinterpret_cast<float *>(static_cast<char *>(ctx->ws) + pb);
    float *P_next = reinterpret_cast<float *>(static_cast<char *>(ctx->ws) + pb + Pb);
    // every machine projects its own gradient; nothing is combined centrally
    const bool one_launch = gossip_step_applies(n);
    if (int rc = ls_gradients_into(ctx, ls, x_dev, ls->G, one_launch ? spread_dev : nullptr)) return rc;
    // then the m-dimensional averaging problem, by gossip with the neighbours: row i is machine i's estimate
    const bool one_group = one_launch && !single_row(n) && project_group(n, ctx->m) >= n;
    const ProjectPlan plan = one_group ? make_project_plan(n, ctx->m, ctx->d, CORE_F32, ctx->sm_count) : ProjectPlan{};
    if (one_group && gossip_joins(n, plan.grid_x)) {
        CORE_CUDA(ctx, launch_project(plan, ctx->keys, ctx->t, ls->G, CORE_F32, n, ls->d, ctx->d, ctx->m, 0, partial, ctx->stream));
        CORE_CUDA(ctx, launch_gossip_step(W_dev, partial, plan.grid_x, nullptr, n, ctx->m, rounds, P_next, reader, spread_dev, ctx->stream));
        P = P_next;
    } else {
        if (int rc = project_all(ctx, ls->G, CORE_F32, n, ls->d, partial, P)) return rc;
        if (one_launch) {
            CORE_CUDA(ctx, launch_gossip_step(W_dev, nullptr, 0, P, n, ctx->m, rounds, P_next, reader, spread_dev, ctx->stream));
            P = P_next;
        } else {
            CORE_CUDA(ctx, launch_gossip_rounds(W_dev, P, n, ctx->m, rounds, P_next, &P, ctx->stream));
            if (spread_dev) CORE_CUDA(ctx, launch_consensus_spread(P, n, ctx->m, reader, spread_dev, ctx->stream));
        }
    }
    // reconstruction from the reader's estimate, update inside the kernel; the printed prefactor n/m is
    // the mean convention's 1/m with an n times longer step
    const ReconstructEpilogue update{x_dev, as_printed ? h * (float)n : h, nullptr, nullptr};
    if (int rc = reconstruct_all(ctx, P + (size_t)reader * ctx->m, x_dev, &update)) return rc;
    ctx->t += 1;
    return CORE_OK;
}

int core_ls_loss(core_ctx *ctx, core_ls *ls, const float *x_dev, double *loss_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !x_dev || !loss_dev || ls->d != ctx->d || ls->device != ctx->device) return CORE_EINVAL;
    return ls_loss_into(ctx, ls, x_dev, loss_dev);
}

int core_ls_loss_host(core_ctx *ctx, core_ls *ls, const float *x_dev, double *loss_host) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!ls || !x_dev || !loss_host || ls->d != ctx->d || ls->device != ctx->device) return CORE_EINVAL;
    if (int rc = ls_loss_into(ctx, ls, x_dev, ls->loss)) return rc;
    CORE_CUDA(ctx, cudaMemcpyAsync(loss_host, ls->loss, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    return CORE_OK;
}

/* ---- run-time diagnostics ------------------------------------------------------ */

int core_debug_force_project_kernel(int kind) {
    if (kind < -1 || kind > 2) return CORE_EINVAL;
    project_force_kernel(kind);
    return CORE_OK;
}

int core_debug_short_kernels(int on) {
    short_kernels_set(on != 0);
    return CORE_OK;
}

int core_debug_fail_allocations(int count) {
    if (count < 0) return CORE_EINVAL;
    g_fail_allocations.store(count);
    return CORE_OK;
}

int core_debug_wait_timeout(uint32_t limit_us, int32_t code, uint32_t observed_host[2]) {
    if (!observed_host || limit_us < 1 || limit_us > 100000 || code < 1) return CORE_EINVAL;
    uint32_t *observed = nullptr;
    if (core_malloc(reinterpret_cast<void **>(&observed), 2 * sizeof(uint32_t)) != cudaSuccess) {
        cudaGetLastError();
        return CORE_ENOMEM;
    }
    cudaError_t e = cudaMemset(observed, 0xFF, 2 * sizeof(uint32_t));
    if (e == cudaSuccess) e = launch_wait_timeout_probe((uint64_t)limit_us * 1000ull, code, observed, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(observed_host, observed, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost);
    cudaFree(observed);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return CORE_ECUDA;
    }
    return CORE_OK;
}

int core_debug_ls_hold_back(core_ls *ls, int32_t chunk) {
    if (!ls || chunk < -1) return CORE_EINVAL;
    ls->step_pass.hold_back = ls->machine_pass.hold_back = chunk < 0 ? INT32_MAX : chunk;
    return CORE_OK;
}

int core_debug_combined_round(core_ctx *ctx, const float *rows_dev, int32_t rows, int64_t ldg, float scale, float *pbar_dev, float *gtilde_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!rows_dev || rows < 1 || ldg < ctx->d || !pbar_dev || !gtilde_dev) return CORE_EINVAL;
    return combined_round(ctx, rows_dev, rows, ldg, scale, pbar_dev, gtilde_dev, nullptr, nullptr);
}

int core_debug_wait_clock(const uint64_t *readings_ns, int32_t count, uint64_t limit_ns, int32_t *given_up_at) {
    if (!readings_ns || !given_up_at || count < 1) return CORE_EINVAL;
    WaitClock clock(readings_ns[0]);
    *given_up_at = -1;
    for (int32_t i = 1; i < count && *given_up_at < 0; ++i)
        if (clock.over(readings_ns[i], limit_ns)) *given_up_at = i;
    return CORE_OK;
}

/* ---- generator windows -------------------------------------------------------- */

int core_debug_philox(core_ctx *ctx, uint32_t j, uint64_t q0, int64_t nq, uint32_t *words_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!words_dev || nq < 0 || (reinterpret_cast<uintptr_t>(words_dev) % 16) != 0) return CORE_EINVAL;
    CORE_CUDA(ctx, launch_debug_philox(ctx->keys, ctx->t, j, q0, nq, words_dev, ctx->stream));
    return CORE_OK;
}

int core_debug_gaussians(core_ctx *ctx, uint32_t j, uint64_t q0, int64_t nq, float *z_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!z_dev || nq < 0 || (reinterpret_cast<uintptr_t>(z_dev) % 16) != 0) return CORE_EINVAL;
    CORE_CUDA(ctx, launch_debug_gaussians(ctx->keys, ctx->t, j, q0, nq, z_dev, ctx->stream));
    return CORE_OK;
}

int core_debug_box_muller(core_ctx *ctx, const uint32_t *words_dev, int64_t nb, float *z_dev) {
    if (int rc = check_ctx(ctx)) return rc;
    if (!words_dev || !z_dev || nb < 0 || (reinterpret_cast<uintptr_t>(words_dev) % 16) != 0 ||
        (reinterpret_cast<uintptr_t>(z_dev) % 16) != 0)
        return CORE_EINVAL;
    CORE_CUDA(ctx, launch_debug_box_muller(words_dev, nb, z_dev, ctx->stream));
    return CORE_OK;
}

int core_debug_project_plan(int32_t n, int32_t m, int64_t d, int dtype, int32_t sm_count, int64_t out[10]) {
    if (!out || n < 1 || m < 1 || d < 1 || sm_count < 1 || !valid_dtype(dtype)) return CORE_EINVAL;
    const ProjectPlan p = make_project_plan(project_group(n, m), m, d, dtype, sm_count);
    const int64_t v[10] = {p.nb, p.jt, p.uq, p.tile_q, p.tj, p.tq, p.grid_x, p.grid_y, p.tiles, (int64_t)p.smem};
    for (int i = 0; i < 10; ++i) out[i] = v[i];
    return CORE_OK;
}

int core_debug_row_plan(int dtype, int32_t rows, int64_t ldg, uint32_t misaligned, int32_t m, int64_t d, int32_t sm_count, int64_t out[10]) {
    if (!out || !valid_dtype(dtype) || rows < 1 || ldg < d || m < 1 || d < 1 || sm_count < 1 || misaligned % elem_size(dtype) != 0) return CORE_EINVAL;
    const void *const G = reinterpret_cast<const void *>(((uintptr_t)1 << 32) + misaligned);      // any address: nothing is read here
    const RowPlan p = make_row_plan(G, dtype, rows, ldg, m, d, sm_count);
    const int64_t v[10] = {p.tile_q, p.tj, p.tq, p.grid_x, p.grid_y, p.tiles, (int64_t)p.smem, p.turn ? 1 : 0, row_plan_columns(m, d, sm_count), p.compute};
    for (int i = 0; i < 10; ++i) out[i] = v[i];
    return CORE_OK;
}

int core_debug_short_plan(int32_t machines, int32_t rows, int32_t m, int64_t d, int32_t sm_count, int64_t out[9]) {
    if (!out || machines < 1 || rows < 1 || m < 1 || d < 1 || sm_count < 1) return CORE_EINVAL;
    const ShortPlan p = make_short_plan(machines, rows, m, d, sm_count), alone = make_short_plan(1, 1, m, d, sm_count);
    const ShortGrid g = alone.ctas > 0 ? make_short_grid(alone, m, d, sm_count, nullptr) : ShortGrid{};
    const int64_t v[9] = {p.ctas, p.per, p.columns, p.lanes, p.slices, (int64_t)p.smem, g.ctas, g.per, g.threads};
    for (int i = 0; i < 9; ++i) out[i] = p.ctas > 0 || i > 5 ? v[i] : 0;
    return CORE_OK;
}

int core_debug_reconstruct_plan(int64_t d, int32_t m, int32_t sm_count, int32_t out[2]) {
    if (!out || d < 1 || m < 1 || sm_count < 1) return CORE_EINVAL;
    out[0] = (int32_t)reconstruct_kernel_for((d + 3) >> 2, m, sm_count);
    const RowPlan row = make_row_plan(nullptr, CORE_F32, 1, d, m, d, sm_count);
    out[1] = reconstruct_joins(row.grid_x, 1, m, d, sm_count) ? 1 : 0;
    return CORE_OK;
}

int core_debug_host_slabs(int64_t d, int32_t n, int dtype, int32_t sm_count, int output, int64_t *lengths, int32_t room, int32_t *count) {
    if (!lengths || !count || d < 1 || n < 1 || !valid_dtype(dtype) || sm_count < 1 || room < 0) return CORE_EINVAL;
    const SlabRule rule = output ? output_slabs(d, sm_count) : input_slabs(d, n, elem_size(dtype));
    *count = 0;
    for (int64_t k0 = 0, len = 0; k0 < d; k0 += len, ++*count) {
        len = next_slab(k0, d, rule);
        if (*count < room) lengths[*count] = len;
    }
    return CORE_OK;
}

int core_debug_ls_reads(int32_t n, int32_t rows, int64_t d, int machines_apart, int32_t sm_count, uint32_t misaligned,
                        int64_t out[3]) {
    if (!out || n < 1 || rows < 1 || d < 1 || sm_count < 1 || misaligned % 4 != 0) return CORE_EINVAL;
    const LsPass pass = make_ls_pass(n, rows, d, machines_apart != 0, sm_count);
    out[0] = pass.units;
    out[1] = out[2] = 0;
    ls_pass_reads(pass, d, ((uintptr_t)1 << 32) + misaligned, &out[1], &out[2]);      // any address: nothing is read here
    return CORE_OK;
}

}  // extern "C"
