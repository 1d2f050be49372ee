// Bulk copies into shared memory that complete on an mbarrier, with bounded
// waits: a wait that runs out (kWaitNs of %globaltimer) returns false, and the
// caller reports it and ends.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gsr {

constexpr uint64_t kWaitNs = 1000000000ull;  // 1 s

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// true when the mbarrier at bar completed the phase with this parity within
// kWaitNs
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    uint32_t done = 0;
    uint64_t t0 = 0;
    for (int it = 0; !done; it++) {
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; "
                     "selp.u32 %0, 1, 0, p; }"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done)
            break;
        if (it == 0)
            t0 = global_ns();
        else if (global_ns() - t0 > kWaitNs)
            return false;
    }
    return true;
}

// late: a test hook, the barrier waits for an arrival that does not come
__device__ __forceinline__ void mbar_init(uint32_t bar, bool late = false)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(late ? 2 : 1) : "memory");
}

__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// dst, src and bytes are multiples of 16
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

}  // namespace gsr
