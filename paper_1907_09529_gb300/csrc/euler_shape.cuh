// euler_shape.cuh -- launch shape of the Euler-Maruyama kernel (lj_euler.cu).  Plain C++ as
// well: the host can compile it alone and check every shape.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define PAMD_HD __host__ __device__
#else
#define PAMD_HD
#endif

namespace pamd {

constexpr int kEulerDense = 192;  // largest N without lists
// Up to this size a particle has eight sums, each over its candidates in increasing j one after
// the other, and double precision takes the library's 1/sqrt; above it two candidates are added
// at a time (single precision), and 1/sqrt is inv_sqrt of lj_math.cuh.  Both are accurate to the
// rounding of the sums (1e-7, 1e-16).  The older order stays where it is as fast, so that small
// paths keep their bits from version to version.
constexpr int kEulerOrdered = 64;
constexpr int kOrderedLg = 3;

// lg: log2 of the partial sums of a particle's force; a thread forms 2^vr of them (the particle
// has 2^(lg - vr) lanes), one after the other, and adds them as the lanes' shuffles would.
struct EulerShape {
    int cs, nloc, lg, vr, nt, cap, npad;
    size_t smem;
};

// First particle of CTA `rank` of the cs <= N that step a chain (rank = cs: N).  Equal shares
// of N / cs, rounded up or down, so that every CTA has particles: with ceil(N / cs) to each,
// 33 particles would leave the last of eight without.
PAMD_HD inline int euler_first(int N, int cs, int rank) { return rank * N / cs; }

// Cluster size, lanes per particle and block size.
// us a step, four chains, with 1, 2, 4, 8 CTAs a chain: N = 32 0.60, 0.70, 0.72, 0.72; N = 48
// 0.78, 0.83, 0.78, 0.79; N = 56 1.05, 0.92, 0.85, 0.85; N = 108 2.4, 1.6, 1.2, 0.98; N = 500
// 13, 7.7, 4.7, 3.5.  So single precision takes clusters from kEulerClusterN particles on, of
// as many CTAs as the chains leave.  Double precision, bound by the FP64 pipe, takes them down
// to four particles each (N = 32: 10.6, 5.9, 5.4, 5.4; N = 64: 39, 20, 10.5, 9.6; N = 108: 110,
// 63, 31, 23).  Chains beyond the SMs get no cluster.
// Partial sums per particle: they set the order of the sums, so they follow from N alone, and a
// chain's path does not depend on the chains beside it or on the GPU: as many as a particle has
// lanes in clusters of eight with about 512 threads (more lanes add shuffles and overhead: N =
// 108 on four CTAs took 1.92 us with 864 threads, 1.78 with 432).  With fewer CTAs a chain a lane
// takes two or four of them, rather than more than 1024 threads, or 512 of more than eight lanes.
// (Lanes by the cluster size instead were up to 1.5 times as fast for 50 chains and more, 96 steps
// of N = 256: 382 us for 50 chains, 529 here, 811 with one CTA of four threads a particle.)
constexpr int kEulerClusterN = 50;
constexpr int kEulerMinLocal = 6;
constexpr int kEulerMinLocalDouble = 4;

inline int euler_lg(int N)
{
    if (N <= kEulerOrdered) return kOrderedLg;
    const int n8 = (N + 7) / 8;
    int lg = 0;
    while (lg < 5 && (n8 << (lg + 1)) <= 512) ++lg;
    return lg;
}

template <typename R>
EulerShape euler_shape(int N, int n_chains, double list_volume, int sms, int max_smem)
{
    constexpr bool F32 = sizeof(R) == 4;
    const int local = F32 ? kEulerMinLocal : kEulerMinLocalDouble;
    EulerShape h;
    h.cs = 1;
    while (h.cs < 8 && (!F32 || N >= kEulerClusterN) && N >= 2 * h.cs * local && 2LL * h.cs * n_chains <= sms) h.cs *= 2;
    h.nloc = (N + h.cs - 1) / h.cs;
    h.lg = euler_lg(N);
    h.vr = 0;
    while (h.vr < 2 && h.vr < h.lg && (h.nloc << (h.lg - h.vr)) > (h.lg - h.vr <= 3 ? 1024 : 512)) ++h.vr;
    const int tpp = 1 << (h.lg - h.vr), sums2 = 2 << h.lg;
    h.nt = std::max(64, (h.nloc * tpp + 31) / 32 * 32);
    const bool list = N > kEulerDense;
    h.npad = (N + sums2 - 1) / sums2 * sums2;
    h.smem = sizeof(R) * (size_t)(list ? 9 : 6) * h.npad;
    h.cap = 0;
    if (list) {  // expected list length plus a margin, every candidate at most, what fits
        const int fit = (int)((max_smem - (long long)h.smem) / (2 * h.nt));
        h.cap = std::max(1, std::min(std::min((N + tpp - 1) / tpp, fit), (int)(1.5 * list_volume / tpp) + 12));
    }
    h.smem = (h.smem + sizeof(uint16_t) * (size_t)h.cap * h.nt + 15) & ~(size_t)15;
    return h;
}

}  // namespace pamd
