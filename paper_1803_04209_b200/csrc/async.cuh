// mbarrier and bulk-copy primitives shared by the kernels that use the asynchronous copy engine.
// Every wait is bounded: it gives up after kWaitLimitNs, records kErrTimeout in the device state
// and tells the rest of the CTA through an abort flag in shared memory.
#pragma once
#include <cstdint>

#include "common.cuh"

namespace cutoff {
namespace async {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// arrive on a barrier given by its shared::cluster address (possibly in another CTA of the cluster).  Relaxed: the
// arrival publishes no memory of this thread (a release at cluster scope would first wait for every earlier global
// store of the warp); callers use it to say "I have finished reading", which their own waits have already ensured.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait.  Gives up after kWaitLimitNs, or soon after another role aborted.  Every lane polls the barrier, the flag and the clock for itself, so
// that lanes may give up at different waits: only for code that goes on in the same way whether the phase is complete or not.
__device__ __forceinline__ void mbar_wait_lane(uint32_t bar, uint32_t parity, volatile int* abort_flag, DevState* st) {
    if (mbar_try_wait(bar, parity)) return;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return;
        if ((it & 7u) == 0u) {                        // a poll of an incomplete phase takes 1.4 us
            if (*abort_flag) return;
            if (global_ns() - t0 > kWaitLimitNs) {
                *abort_flag = 1;
                atomicOr(&st->error_flags, kErrTimeout);
                return;
            }
        }
    }
}

// Bounded wait of a whole warp.  Returns false, in all lanes, if it gave up or if another role already aborted: an election, a warp barrier or a
// tensor-memory access takes all lanes, so lanes that part ways on the result could wait for one another without a limit.  (A
// vote on every poll: one vote behind polls of every lane is slower, emission at N = 1024, S = 65536 116.7 us against 115.1.)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, DevState* st) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 1;; ++it) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if ((it & 63u) == 0u) {
            if (__any_sync(0xffffffffu, *abort_flag)) return false;
            if (__any_sync(0xffffffffu, global_ns() - t0 > kWaitLimitNs)) {
                *abort_flag = 1;
                atomicOr(&st->error_flags, kErrTimeout);
                return false;
            }
        }
    }
}

// 1-D bulk copy global -> shared; bytes, source and destination are multiples of 16.
__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// Plain bounded wait for wind-down paths (no flag, no error record).
__device__ __forceinline__ void mbar_wait_quiet(uint32_t bar, uint32_t parity) {
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity) && global_ns() - t0 < kWaitLimitNs) {}
}

}  // namespace async
}  // namespace cutoff
