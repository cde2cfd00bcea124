// ea_async.cuh -- shared-memory staging primitives for sm_103a (inline PTX): mbarriers, the bulk
// (TMA, one-dimensional, no multicast) global->shared copy, 4-byte cp.async completing on an
// mbarrier, and waits with a time limit.
//
// A wait that exceeds its limit returns false; the caller records EA_STATUS_TIMEOUT in the
// workspace status word (read by ea_sync_status) and stops, after draining its own copies.
#pragma once

#include <cstdint>
#include <utility>

#include <cuda_runtime.h>

namespace ea {

constexpr uint32_t kStatusTimeout = 1u;
constexpr uint32_t kStatusCheck = 2u;  // a kernel found an input outside what its launch assumed
constexpr long long kWaitLimitCycles = 4000000000LL;  // ~2 s at the 2.07 GHz SM clock

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// Make barrier initialisation visible to the async (copy) proxy before first use.
__device__ __forceinline__ void mbar_init_fence()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Order this thread's plain accesses to shared memory before later ones of the async (copy) proxy, which
// an mbarrier alone does not: the reader of a stage that a bulk copy refills calls it before it arrives
// on the stage's barrier, if it has also written there.
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase with the given parity to complete; false after ~2 s.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit_cycles = kWaitLimitCycles)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > limit_cycles) return false;
    return true;
}

// Bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned) from global memory to this
// CTA's shared memory; completion is counted on `bar` as transaction bytes.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

// 4-byte asynchronous copy global -> shared (cached at all levels).
__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// 16-byte asynchronous copy global -> shared (both addresses 16-byte aligned; cached in L2 only).
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Wait until every cp.async this thread issued has landed in shared memory.
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One arrival on `bar` once every cp.async this thread issued before has landed (the barrier's
// expected count already includes it).
__device__ __forceinline__ void cp_async_arrive_noinc(uint64_t *bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void report_status(uint32_t *status, uint32_t code)
{
    if (status) atomicOr(status, code);
}

// Programmatic dependent launch.  The round's kernels are launched with programmatic stream
// serialization (launch_pdl): each lets the next kernel on the stream be scheduled as soon as all of
// its own CTAs have started (pdl_trigger), and each waits, before its first access to anything that a
// kernel writes, until the previous kernel has completed and its writes are visible (pdl_wait).  The
// next kernel's launch, shared-memory prologue and lookups in the handle's constant tables thus
// overlap this one's last CTAs; the data order of the stream is unchanged.  Without the launch attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// How an SM's 256 KB are split between L1 and shared memory, as a percentage of the largest shared
// memory (228 KB): 44 asks for 100 KB, which holds the resident CTAs of every kernel but the staged
// and grouped ones.  The rest is L1, where every load in flight takes its line: 8 TB/s at ~0.8 us is
// ~40 KB of reads in flight per SM, more than the 28 KB that the largest split leaves.
constexpr int kCarveoutPercent = 44;

// Launch `kernel` with programmatic stream serialization (see pdl_trigger / pdl_wait), or, with
// overlap = false, after everything before it on the stream has finished.
//
// An SM changes its split only when it is empty, and dependent launches fill it with the next
// kernel's CTAs before the last one's have left, so a split stays as long as the chain does.  The
// kernels of a chain therefore ask for the same one, and the first kernel after a staged or grouped
// server, which run at the largest, is launched with overlap = false (the caller's job).  With the
// driver's own choice, rounds queued one behind another ran their worker passes at the server's
// split: 17.73 ms at d = 400,000,007, n = 8 (1-bit 4096-blocks), where a round on its own took
// 14.02 ms; every kernel at the largest split measured 18.27 ms.
template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool overlap,
                       int carveout, Args &&...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[0].val.sharedMemCarveout = carveout;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace ea
