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
// Up to this size a particle has eight lanes, each adding its candidates in increasing j, and
// double precision takes the library's 1/sqrt: the arithmetic of the LJ kernels' plain form,
// bit for bit.  Small boxes are where a start can overlap (33 to 45 particles on a lattice of
// 108 sites), and such a path turns any other order of the sums into another path.
constexpr int kEulerOrdered = 64;
constexpr int kOrderedLg = 3;

struct EulerShape {
    int cs, nloc, lg, nt, cap, npad;
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
// Lanes per particle: about 512 threads (more lanes add shuffles and overhead: N = 108 on four
// CTAs took 1.92 us with 864 threads, 1.78 with 432), up to 1024 where that keeps four lanes.
constexpr int kEulerClusterN = 50;
constexpr int kEulerMinLocal = 6;
constexpr int kEulerMinLocalDouble = 4;

template <typename R>
EulerShape euler_shape(int N, int n_chains, double list_volume, int sms, int max_smem)
{
    constexpr bool F32 = sizeof(R) == 4;
    const int local = F32 ? kEulerMinLocal : kEulerMinLocalDouble;
    EulerShape h;
    h.cs = 1;
    while (h.cs < 8 && (!F32 || N >= kEulerClusterN) && N >= 2 * h.cs * local && 2LL * h.cs * n_chains <= sms) h.cs *= 2;
    h.nloc = (N + h.cs - 1) / h.cs;
    h.lg = 0;
    if (N <= kEulerOrdered)
        h.lg = kOrderedLg;
    else
        while (h.lg < 5 && (h.nloc << (h.lg + 1)) <= (h.lg < 2 ? 1024 : 512)) ++h.lg;
    h.nt = std::max(64, ((h.nloc << h.lg) + 31) / 32 * 32);
    const int tpp = 1 << h.lg;
    const bool list = N > kEulerDense;
    h.npad = (N + 2 * tpp - 1) / (2 * tpp) * (2 * tpp);
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
