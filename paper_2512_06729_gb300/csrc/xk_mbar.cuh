// Exchange between the CTAs of a cluster: addresses in another CTA's shared memory, and mbarriers that
// count what arrives there.
#pragma once

#include <stdint.h>

#include "xk_internal.cuh"

namespace xk {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_init(uint32_t bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bounded wait for a phase, as the other waits on CTAs: ctl->wait_polls polls (kSyncPolls unless set)
// or until another wait has given up.  A try_wait sleeps up to 4 us by itself and counts as kTryPolls; the
// limit is looked up once the first has come back empty (fetched before it, it was on the chain of every
// column: eight steps of 20 species took 2.67 ms instead of 2.49).  Giving up is recorded, and the caller
// carries on (every index it takes from what did not arrive is clamped) to the barrier where its cluster
// leaves together.
constexpr unsigned kTryPolls = 32;
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, Ctl *ctl)
{
    unsigned long long limit = kTryPolls;
    for (unsigned long long i = 0; i < limit; i += kTryPolls) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return;
        if (i == 0) limit = ctl->wait_polls ? ctl->wait_polls : kSyncPolls;
        if (*(volatile int *)&ctl->err_timeout) return;
    }
    atomicExch(&ctl->err_timeout, 1);
}

}  // namespace xk
