// Bulk asynchronous global -> shared copies completed on shared-memory mbarriers.
//
// One elected thread arms a barrier with the byte count it expects and issues
// cp.async.bulk copies that signal the barrier as they land; consumers wait on the
// barrier's phase parity.  Every wait is bounded in time (%globaltimer): a wait that runs
// out returns false so that the kernel can raise an error flag and leave instead of
// hanging the device.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace wcsim {

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s: far above any legitimate wait
constexpr int kErrInvalidDepo = 1;                 // device flag bits
constexpr int kErrTimeout = 2;

// First statement (after work on this CTA's own shared memory and on data that never changes) of
// every kernel launched with launch_chained, by every thread of it: waits until the kernel before
// it on the stream has completed and its writes are visible, then lets the next one be put on the
// SMs.  No CTA may leave before it: the next kernel takes this one's completion for that of
// everything earlier.
__device__ __forceinline__ void after_previous_kernel()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads of what the kernel before this one wrote: ordinary ones, kept behind
// after_previous_kernel().  The read-only path (__ldg, or a plain read through a const __restrict__
// pointer) is for data that does not change while a kernel is on the SMs, and the compiler may move
// such loads across anything.
__device__ __forceinline__ float2 ld_fresh(const float2* p)
{
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

// Make barrier initialisation visible to the async proxy before first use.
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Order this thread's earlier shared-memory accesses before later async-proxy writes.
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// dst (shared) <- src (global), `bytes` a multiple of 16, both addresses 16-byte aligned.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Hint: bring `bytes` (a multiple of 16) of global memory at p (16-byte aligned, inside one
// allocation) into L2 without waiting; later loads of the range then hit L2.
__device__ __forceinline__ void bulk_prefetch_l2(const void* p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Tensor store: the box of the 5-D tensor map at `map` (a kernel parameter) whose first
// element has coordinates (c0 .. c4) <- shared memory at src (128-byte aligned, the box in
// dense order).  Completion is tracked by bulk groups (bulk_commit / bulk_wait_read).
__device__ __forceinline__ void tma_store_5d(const void* map, const void* src, int c0, int c1,
                                             int c2, int c3, int c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];"
        ::"l"(map), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

__device__ __forceinline__ void bulk_commit()
{
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Wait until every committed bulk group of this thread has finished reading shared memory
// (the source may then be reused or released).
__device__ __forceinline__ void bulk_wait_read()
{
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
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

// Non-blocking test of the phase with the given parity.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait until the barrier's phase with the given parity completes; false once limit_ns has
// passed (the clock is checked before each potentially suspending try_wait, so a limit of 0
// gives one non-blocking test).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          uint64_t limit_ns = kWaitLimitNs)
{
    if (mbar_test_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (;;) {
        if (globaltimer_ns() - t0 >= limit_ns) return false;
        if (mbar_try_wait(bar, parity)) return true;
    }
}

}  // namespace wcsim
