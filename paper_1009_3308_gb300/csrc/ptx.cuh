// Inline-PTX helpers for sm_103a: mbarriers, bulk async copies (TMA engine,
// 1-D form), L2 cache policies.  Every wait is bounded: after
// SPH_WAIT_LIMIT polls it records a timeout in the CTA's abort flag (and in
// the plan's device status word) and returns false, so that no kernel can
// spin forever.
#pragma once
#include <cstdint>

namespace sph {

#ifndef SPH_WAIT_LIMIT
#define SPH_WAIT_LIMIT (1u << 26)
#endif

// device status word bits
#define SPH_STATUS_TIMEOUT 1u

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// make barrier initialisation visible to the async (TMA) proxy
__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of the given parity.  abort: CTA-shared flag;
// once set, waits return false immediately.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                          unsigned* status) {
    for (uint32_t i = 0; i < SPH_WAIT_LIMIT; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort) return false;
    }
    *abort = 1;
    if (status) atomicOr(status, SPH_STATUS_TIMEOUT);
    return false;
}

// Bounded wait at the end of a role for what it has in flight, bulk copies into the
// CTA's shared memory or MMAs on its tensor memory: these finish by themselves, so
// it goes on when abort is set (the CTA must not exit under them), for a time that
// no copy or MMA takes.
__device__ __forceinline__ bool mbar_drain(uint64_t* bar, uint32_t parity, unsigned* status) {
    constexpr uint32_t limit = SPH_WAIT_LIMIT < (1u << 16) ? SPH_WAIT_LIMIT : 1u << 16;
    for (uint32_t i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    if (status) atomicOr(status, SPH_STATUS_TIMEOUT);
    return false;
}

// mbar_wait for two barriers: both are polled before either result is used (a
// poll that succeeds at once takes 150 to 200 cycles in a busy CTA).
__device__ __forceinline__ bool mbar_wait2(uint64_t* bar0, uint32_t parity0, uint64_t* bar1, uint32_t parity1,
                                           volatile int* abort, unsigned* status) {
    for (uint32_t i = 0; i < SPH_WAIT_LIMIT; ++i) {
        const bool r0 = mbar_try_wait(bar0, parity0), r1 = mbar_try_wait(bar1, parity1);
        if (r0 && r1) return true;
        if (*abort) return false;
    }
    *abort = 1;
    if (status) atomicOr(status, SPH_STATUS_TIMEOUT);
    return false;
}

// L2 policy: evict-first (streamed-once table data must not displace the
// L2-resident intermediates)
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// L2 policy: evict-last (small operands re-read by several CTAs or stages)
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// 1-D bulk copy global -> shared (dst, src 16-byte aligned; bytes % 16 == 0),
// completion counted on the mbarrier as transaction bytes.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                         uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1], %2, [%3], %4;" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialisation may start while its predecessor drains; pdl_wait() blocks the
// calling thread until the predecessor grid has completed and its writes are
// visible (a no-op for a normal launch), pdl_launch() lets the successor grid
// start its prologue.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void named_bar_sync(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

}  // namespace sph
