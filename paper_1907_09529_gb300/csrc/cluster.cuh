// cluster.cuh -- exchange between the CTAs of a thread-block cluster.  Values travel as
// asynchronous stores that a transaction barrier (mbarrier) of the receiving CTA counts:
// nobody waits for an acknowledgement, and a CTA goes on as soon as the bytes of its own copy
// are there.  Remote stores and a cluster barrier take about 0.4 us longer a round, most of
// it the release waiting for the stores.
#pragma once

#include "pamd_internal.cuh"

namespace pamd {

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned shared_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned remote_addr(unsigned a, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void send_async(unsigned to, float v, unsigned bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(to),
                 "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send_async(unsigned to, double v, unsigned bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(to),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void barrier_init(unsigned bar)  // one arrival a phase
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void barrier_init_done()  // (before a cluster barrier)
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// One phase of a barrier: `bytes` of asynchronous stores, and this call.
__device__ __forceinline__ void expect(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool phase_done(unsigned bar, unsigned parity)
{
    unsigned done;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return done != 0;
}
__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Waits for the phase of the given parity; false when it did not complete within two seconds.
__device__ __forceinline__ bool wait_phase(unsigned bar, unsigned parity)
{
    if (phase_done(bar, parity)) return true;
    const unsigned long long end = now_ns() + 2000000000ull;
    while (!phase_done(bar, parity))
        if (now_ns() > end) return false;
    return true;
}

}  // namespace pamd
