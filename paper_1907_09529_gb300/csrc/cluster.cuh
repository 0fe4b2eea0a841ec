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
// The limit of a launch's waits: `ns` of time, twice, so that a wait does not run out because the
// process was stopped for a while.  Tests make waits run out: the odd CTAs of a cluster leave
// after `rounds` rounds.
struct WaitLimit {
    unsigned ns = 2000000000u;
    int rounds = 0x7fffffff;
};

// Waits for the phase of the given parity; false when the wait ran out.
__device__ __forceinline__ bool poll_phase(unsigned bar, unsigned parity, unsigned ns)
{
    const unsigned long long end = now_ns() + ns;
    while (!phase_done(bar, parity))
        if (now_ns() > end) return false;
    return true;
}
__device__ __forceinline__ bool wait_phase(unsigned bar, unsigned parity, const WaitLimit& w)
{
    return poll_phase(bar, parity, w.ns) || poll_phase(bar, parity, w.ns);
}

// How the CTAs of a cluster part: in shared memory, cleared before the first cluster barrier.
struct ClusterEnd {
    unsigned lost;       // some wait of the cluster ran out
    unsigned out[8][2];  // bytes this CTA sent to the barriers of every CTA
    unsigned in[8][2];   // bytes every CTA sent to this one's
};

__device__ __forceinline__ void put_remote(unsigned* p, unsigned rank, unsigned v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote_addr(shared_addr(p), rank)), "r"(v) : "memory");
}
// Takes `bytes` off what a barrier's phase waits for, as if they had arrived.
__device__ __forceinline__ void complete_bytes(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Called by every thread of a cluster after its last round, with `lost` where a wait ran out
// (that thread has sent and armed nothing since).  False: nothing was lost, and since every phase
// was waited for, no store is under way.  True, for every thread of the cluster: some wait ran
// out, and cluster_drain has to follow.
__device__ __forceinline__ bool cluster_lost(ClusterEnd* E, bool lost, int cs)
{
    if (__syncthreads_or(lost) && threadIdx.x < cs) put_remote(&E->lost, threadIdx.x, 1u);
    cluster_barrier();  // (no CTA sends any more)
    return *reinterpret_cast<volatile unsigned*>(&E->lost) != 0u;
}

// After a lost wait stores may still be under way to CTAs that wait for nothing any more, and a
// CTA must not end before they have landed.  `count` adds up in E->out what this CTA has sent
// (called by every thread); phases(b) of `bytes` each were armed on barrier b.  With what every
// CTA has sent known, each barrier is made to wait for just that.
template <typename Phases, typename Count>
__device__ __forceinline__ void cluster_drain(ClusterEnd* E, unsigned bar0, unsigned bytes, int cs, Phases&& phases,
                                              Count&& count)
{
    const int tid = threadIdx.x;
    const unsigned rank = cluster_rank();
    count();
    __syncthreads();
    if (tid < 2 * cs) put_remote(&E->in[rank][tid & 1], (unsigned)tid >> 1, E->out[tid >> 1][tid & 1]);
    cluster_barrier();
    if (tid < 2) {
        const unsigned bar = bar0 + 8u * (unsigned)tid, n = phases(tid);
        unsigned sent = 0;
        for (int r = 0; r < cs; ++r) sent += E->in[r][tid];
        const int missing = (int)(n * bytes - sent);  // (below 2^20 in size: differences of the last phases)
        if (missing > 0) complete_bytes(bar, (unsigned)missing);
        bool there = n == 0 || wait_phase(bar, (n - 1) & 1u, WaitLimit());
        if (missing < 0 && there) {  // bytes of a phase that was not armed
            expect(bar, (unsigned)-missing);
            wait_phase(bar, n & 1u, WaitLimit());
        }
    }
    __syncthreads();
    cluster_barrier();
}

}  // namespace pamd
