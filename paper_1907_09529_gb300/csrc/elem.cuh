// elem.cuh -- the order in which a block of kElemThreads threads visits the elements of an
// ElemBlock in the element-wise kernels.  Per-thread sums are taken in this order, so the
// kernels that must agree bit for bit share it.
//
// Single precision: the aligned float4s of the buffer inside the block (thread t takes
// vectors t, t + 256, ...), then the at most 3 + 3 elements before and after them, one per
// thread.  A chain need not start on a 16-byte boundary (with an odd number of elements
// per chain three chains in four do not), so the vectors are those of the buffer, not of
// the chain.  Double precision: element t, t + 256, ...
#pragma once

#include "pamd_internal.cuh"

namespace pamd {

template <typename R>
struct ElemOrder;

template <>
struct ElemOrder<float> {
    int head, nvec, nbody, tail;  // elements before the first vector, vectors, after the last
    __device__ __forceinline__ explicit ElemOrder(const ElemBlock& B)
    {
        head = min(B.n, (int)((4 - ((B.chain_base + B.e0) & 3)) & 3));
        nvec = (B.n - head) >> 2;
        nbody = 4 * nvec;
        tail = B.n - head - nbody;
    }
    __device__ __forceinline__ bool vec(int k) const { return (int)threadIdx.x + k * kElemThreads < nvec; }
    __device__ __forceinline__ int rel(int k) const { return head + 4 * ((int)threadIdx.x + k * kElemThreads); }
    __device__ __forceinline__ bool one(int k) const { return k == 0 && (int)threadIdx.x < head + tail; }
    __device__ __forceinline__ int rel1(int) const
    {
        return (int)threadIdx.x < head ? (int)threadIdx.x : nbody + (int)threadIdx.x;
    }
};

template <>
struct ElemOrder<double> {
    int n;
    __device__ __forceinline__ explicit ElemOrder(const ElemBlock& B) : n(B.n) {}
    __device__ __forceinline__ bool vec(int) const { return false; }
    __device__ __forceinline__ int rel(int) const { return 0; }
    __device__ __forceinline__ bool one(int k) const { return (int)threadIdx.x + k * kElemThreads < n; }
    __device__ __forceinline__ int rel1(int k) const { return (int)threadIdx.x + k * kElemThreads; }
};

// zs[q..q+3] for any q from two aligned 16-byte loads (zs 16-byte aligned, readable to
// the end of the vector that holds q + 3).  The offset q & 3 is the same for a whole block.
__device__ __forceinline__ float4 unaligned4(const float* zs, int q)
{
    const float4 a = *reinterpret_cast<const float4*>(zs + (q & ~3));
    const int o = q & 3;
    if (o == 0) return a;
    const float4 b = *reinterpret_cast<const float4*>(zs + (q & ~3) + 4);
    if (o == 1) return make_float4(a.y, a.z, a.w, b.x);
    if (o == 2) return make_float4(a.z, a.w, b.x, b.y);
    return make_float4(a.w, b.x, b.y, b.z);
}

// Metropolis-Hastings test of one chain from its sums.
__device__ __forceinline__ int mala_decide(int c, double S, double S_prop, double qf, double qr,
                                           const double* log_u, const MalaDev& md, int update_index,
                                           double* log_alpha)
{
    const double h4 = 4.0 * md.h;
    const double la = (S - S_prop) - qr / h4 + qf / h4;
    const double lu = log_u ? log_u[c]
                            : log(philox_uniform53(md.seed, md.counter + (uint64_t)update_index, kStreamAccept,
                                                   (uint32_t)c));
    if (log_alpha) log_alpha[c] = la;
    return (lu < la) ? 1 : 0;  // NaN log alpha never accepts
}

}  // namespace pamd
