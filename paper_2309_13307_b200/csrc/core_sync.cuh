// Thin wrappers over the PTX for barriers in shared memory and bulk copies, shared by the kernels that hand
// buffers over with them.  Every wait is bounded by the device's global timer.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace core {

// A kernel of a chain (launch_chained): until everything before it in the stream is done and visible ...
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// ... and from here on the kernel after it may be scheduled where there is room (it waits in turn).
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr uint64_t kWaitLimitNs = 100ull * 1000 * 1000;   // a wait gives up after 100 ms

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One arrival that also announces `bytes` of asynchronous copies or stores to this barrier.
__device__ __forceinline__ void mbar_arrive_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Announces `bytes` more without arriving.
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Time spent waiting, from readings of the global timer.  That timer runs on while the GPU works for somebody else (time
// slices, a debugger), so what lies between two readings counts kWaitStepNs at most: a wait is given up for the time its
// program was there to be served, not for the time it was away.
constexpr uint64_t kWaitStepNs = 1000ull * 1000;          // 1 ms; eight probes take some microseconds
struct WaitClock {
    uint64_t last, spent = 0;
    __host__ __device__ explicit WaitClock(uint64_t now) : last(now) {}
    __host__ __device__ bool over(uint64_t now, uint64_t limit_ns) {
        spent += now - last < kWaitStepNs ? now - last : kWaitStepNs;
        last = now;
        return spent >= limit_ns;
    }
};
// Bounded wait: false when the phase did not complete within limit_ns (see WaitClock).  The timer is read only
// once a number of probes have failed (a probe waits for a while by itself): a wait for memory is normally served
// long before.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns = kWaitLimitNs) {
#pragma unroll 1
    for (int probe = 0; probe < 64; ++probe)
        if (mbar_try_wait(bar, parity)) return true;
    WaitClock clock(global_timer_ns());
    do {
#pragma unroll 1
        for (int probe = 0; probe < 8; ++probe)
            if (mbar_try_wait(bar, parity)) return true;
    } while (!clock.over(global_timer_ns(), limit_ns));
    return false;
}
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// L2 policy of data that makes way first.
__device__ __forceinline__ uint64_t l2_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// Asks for `bytes` (a multiple of 16, 16-byte aligned) to be brought into L2: a hint, nothing is read by the program.
__device__ __forceinline__ void bulk_prefetch(const void *gmem_src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(gmem_src), "r"(bytes) : "memory");
}
// `bytes` (a multiple of 16) from global to shared memory, both 16-byte aligned; completion is counted on `bar`.
__device__ __forceinline__ void bulk_copy(uint32_t smem_dst, const void *gmem_src, uint32_t bytes, uint32_t bar, uint64_t policy) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(smem_dst),
                 "l"(gmem_src), "r"(bytes), "r"(bar), "l"(policy)
                 : "memory");
}

// Thread-block clusters: this CTA's rank, the barrier over all threads of the cluster that have not exited, in two halves, and a store to
// the same place of another CTA's shared memory (which has to have started: one barrier before the first such store).
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void store_remote(const float *smem, uint32_t rank, float v) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(smem)), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
}

__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int threads) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

}  // namespace core
