// lj_euler.cu -- Euler-Maruyama paths of Lennard-Jones systems (Eq. (2)):
//   x_{t+1} = x_t + a F(x_t) + sqrt(2 D dt) xi_t,  each new slice stored in the
// path's precision and used as stored.
//
// What bounds it: the serial chain of steps.  A step's forces need every position of
// the step before, so only the work inside one step can be spread, and what counts is the
// latency of a step.
//   * The normals do not depend on the path: a kernel over all elements first writes them
//     into the slices that the steps will overwrite (slice t + 1 holds xi_t), and a step
//     loads its own two steps ahead.  Drawing them inside the step put ten Philox rounds
//     and Box-Muller on the chain.
//   * A chain is stepped by a cluster of CTAs (up to 8).  Each CTA holds all positions
//     and moves N / CS particles, up to 32 lanes to a particle (how many partial sums a force
//     has, and so every bit of a path, follows from N alone: euler_shape.cuh); the new
//     coordinates go to every CTA's shared memory as asynchronous stores counted by a
//     transaction barrier there.  A step costs one trip between SMs; with plain remote stores
//     and a cluster barrier it also waited for their acknowledgement (N = 108: 1.33 against
//     0.96 us a step).  Waits are bounded; what follows one that runs out is in cluster.cuh.
//   * Small systems (N <= kEulerDense) evaluate every pair: no list, no displacement check,
//     two candidates per packed f32x2 operation.  Larger ones walk Verlet lists of radius
//     rc + skin, rebuilt when some particle has moved skin / 2 (a list that overflows scans
//     all candidates).
// N = 108, four chains of 1024 steps: 4.89 ms (4.8 us a step) with one CTA of four threads
// per particle and the normals in the step, 0.96 ms (0.94 us) now; a step of N = 500, eight
// chains, 17.5 -> 3.4 us, of N = 108 in double precision 101 -> 23 us.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cluster.cuh"
#include "euler_shape.cuh"
#include "lj_math.cuh"

namespace pamd {

namespace {

// The normals of every element of slices 1..T of a system's chains, into the path.
template <typename R>
__global__ void euler_normals_kernel(R* __restrict__ pos, long long off, long long chain_len, int s,
                                     int chain0, uint64_t seed, uint64_t counter)
{
    const int b = blockIdx.x;
    R* X = pos + off + (long long)b * chain_len;
    const long long ng = (chain_len + 3) >> 2, g0 = s >> 2;
    for (long long g = g0 + (long long)blockIdx.y * blockDim.x + threadIdx.x; g < ng;
         g += (long long)gridDim.y * blockDim.x) {
        const float4 z = philox_normals4(seed, counter, kStreamEuler, (uint32_t)(chain0 + b), (uint32_t)g);
        const float v[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const long long e = 4 * g + l;
            if (e >= s && e < chain_len && PAMD_OK_IDX(e, chain_len)) X[e] = (R)v[l];
        }
    }
}

// Positions of one slice in shared memory.  Single precision, no list: candidates 2k and
// 2k + 1 of lane q (j = q + tpp m) form one float2 per component.  Otherwise three arrays.
template <typename R, bool LIST>
struct EulerPos {
    R* p;
    int n, lg;  // padded particles; log2 of the partial sums per particle
    __device__ __forceinline__ R* at(int j, int c) const
    {
        if (sizeof(R) == 4 && !LIST) {  // (LG >= 0)
            const int m = j >> lg, q = j & ((1 << lg) - 1);
            return p + c * n + (((m >> 1) << lg) + q) * 2 + (m & 1);
        }
        return p + c * n + j;
    }
};

// Force on a particle from a lane's candidates, every pair, two per packed operation; the
// constants are set up once, outside the steps.
template <int LG>
struct DenseForce {
    float2 nL, iL, mag, nmag, c1, c2, m1, duc;
    float rc2;
    int N, full, all, i, py, pz;
    __device__ __forceinline__ DenseForce(const LJK<float>& k, int N_, int npad, int i_)
        : nL(pk(-k.L)), iL(pk(k.iL)), mag(pk(12582912.0f)), nmag(pk(-12582912.0f)), c1(pk(k.c1)), c2(pk(k.c2)),
          m1(pk(-1.0f)), duc(pk(k.duc)), rc2(k.rc2), N(N_), full(N_ >> (LG + 1)), all(npad >> (LG + 1)), i(i_),
          py(npad / 2), pz(npad)
    {
    }
    template <bool CHECK>
    __device__ __forceinline__ void two(const float2* a, int j, float2 x, float2 y, float2 z, float2& fx, float2& fy,
                                        float2& fz) const
    {
        const int j2 = j + (1 << LG);
        const float inf = __int_as_float(0x7f800000);
        float2 dx = sub2(x, a[0]), dy = sub2(y, a[py]), dz = sub2(z, a[pz]);
        dx = fma2(nL, add2(fma2(dx, iL, mag), nmag), dx);
        dy = fma2(nL, add2(fma2(dy, iL, mag), nmag), dy);
        dz = fma2(nL, add2(fma2(dz, iL, mag), nmag), dz);
        float2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        // r^2 = +inf: exact zeros (outside the cutoff, itself, padding)
        r2.x = (r2.x <= rc2 && j != i && (!CHECK || j < N)) ? r2.x : inf;
        r2.y = (r2.y <= rc2 && j2 != i && (!CHECK || j2 < N)) ? r2.y : inf;
        const float2 ri = pk(inv_sqrt(r2.x), inv_sqrt(r2.y)), ir2 = mul2(ri, ri);
        const float2 ir6 = mul2(mul2(ir2, ir2), ir2), u = mul2(c1, ir6), t = fma2(c2, ir6, m1);
        const float2 fs = fma2(mul2(u, t), ir2, mul2(duc, ri));
        if (LG == kOrderedLg) {  // one sum, in increasing j
            fx.x = fma_r(fs.y, dx.y, fma_r(fs.x, dx.x, fx.x));
            fy.x = fma_r(fs.y, dy.y, fma_r(fs.x, dy.x, fy.x));
            fz.x = fma_r(fs.y, dz.y, fma_r(fs.x, dz.x, fz.x));
        } else {
            fx = fma2(fs, dx, fx);
            fy = fma2(fs, dy, fy);
            fz = fma2(fs, dz, fz);
        }
    }
    // p: the slice; candidates 2m, 2m + 1 of sum q are the float2 at m 2^LG + q.  SKIP: nothing
    // is done for a last pair of padding (exact zeros): for lanes with several sums, where it
    // is worth the test (200 chains of N = 65: 3.5 against 4.4 us a step)
    template <bool SKIP>
    __device__ __forceinline__ void sum(const float* p, const float (&xi)[3], int q, float (&f)[3]) const
    {
        const float2 x = pk(xi[0]), y = pk(xi[1]), z = pk(xi[2]);
        float2 fx = pk(0.0f), fy = pk(0.0f), fz = pk(0.0f);
        const float2* a = reinterpret_cast<const float2*>(p) + q;
        int j = q;
#pragma unroll 2
        for (int m = 0; m < full; ++m, j += 2 << LG, a += 1 << LG) two<false>(a, j, x, y, z, fx, fy, fz);
        if (full < all && (!SKIP || j < N)) two<true>(a, j, x, y, z, fx, fy, fz);
        f[0] = fx.x + fx.y;
        f[1] = fy.x + fy.y;
        f[2] = fz.x + fz.y;
    }
};

__device__ __forceinline__ const LJK<float>& dense_consts(const LJK<float>& k) { return k; }
__device__ __forceinline__ LJK<float> dense_consts(const LJK<double>&) { return LJK<float>(); }  // (not used)

// Lanes 0..2 of a particle (one lane when it has fewer) take its components x, y, z; lane
// q writes component q mod 3 of the new position to CTAs q / 3, q / 3 + tpp / 3, ...
struct EulerLane {
    int comp, first, stride, nc;  // nc: components of a mover lane
    bool mover, owner;            // of a lane of a particle
    __device__ __forceinline__ EulerLane(int q, int tpp, bool active)
    {
        const int lanes3 = tpp / 3;
        comp = tpp >= 3 ? q % 3 : 0, first = tpp >= 3 ? q / 3 : 0, stride = tpp >= 3 ? lanes3 : 1, nc = tpp >= 3 ? 1 : 3;
        mover = active && (tpp >= 3 ? q < 3 * lanes3 : q == 0), owner = mover && q < 3;
    }
};

// After a lost wait of a cluster; a thread has sent slices 1..sent[tid].  The chain is left as
// NaN after slice 0: what it holds by then, normals among it, looks like positions.  (Not inlined:
// what it needs would be kept in registers throughout the steps.)
template <typename R>
__device__ __noinline__ void euler_drain(ClusterEnd* E, const int* sent, unsigned bar0, int N, int T, int cs, int lanes,
                                         R* X)
{
    const int rank = (int)cluster_rank(), tid = threadIdx.x;
    auto count = [&] {
        const int mine = euler_first(N, cs, rank + 1) - euler_first(N, cs, rank);
        const EulerLane l(tid & ((1 << lanes) - 1), 1 << lanes, (tid >> lanes) < mine);
        for (int d = l.first; l.mover && d < cs; d += l.stride) {
            atomicAdd(&E->out[d][0], (unsigned)(sent[tid] / 2) * (unsigned)(l.nc * sizeof(R)));
            atomicAdd(&E->out[d][1], (unsigned)((sent[tid] + 1) / 2) * (unsigned)(l.nc * sizeof(R)));
        }
    };
    // slices 1..armed: 1 and 2 to begin with, t + 2 in step t
    auto phases = [&](int b) { return (unsigned)((min(T, max(sent[0] + 1, 2)) + b) / 2); };
    cluster_drain(E, bar0, (unsigned)(3 * N * sizeof(R)), cs, phases, count);
    const long long s = 3 * N, n = (long long)(T + 1) * s;
    for (long long e = s + (long long)rank * blockDim.x + tid; e < n; e += (long long)cs * blockDim.x)
        if (PAMD_OK_IDX(e, n)) X[e] = (R)__int_as_float(0x7fffffff);
}

// f = the sum over s = V, V + W, ... of the partial sums `leaf(s, f)` (S of them in all), as the
// shuffles of lanes s would add them: first s and s + S/2, then s and s + S/4, ...
template <typename R, int V, int W, int S, typename F>
__device__ __forceinline__ void sum_tree(R (&f)[3], F&& leaf)
{
    if constexpr (W == S) {
        leaf(std::integral_constant<int, V>{}, f);
    } else {
        R g[3];
        sum_tree<R, V, 2 * W, S>(f, leaf);
        sum_tree<R, V + W, 2 * W, S>(g, leaf);
#pragma unroll
        for (int c = 0; c < 3; ++c) f[c] += g[c];
    }
}

// LG: log2 of the partial sums per particle where it is known (the all-pairs form), else -1; a
// lane takes 2^VR of them.
template <typename R, bool LIST, int LG, int VR, int MAXT>
__global__ void __launch_bounds__(MAXT)
    lj_euler_kernel(R* __restrict__ pos, const R* __restrict__ noise, const LJSysDev<R> S, const EulerShape H,
                    int* __restrict__ err, const WaitLimit limit)
{
    extern __shared__ __align__(32) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_bar[2];  // of the two slices
    // Behind the arrays of the steps: as static shared memory, in front of them, these two made a
    // step of N = 108 take 8 to 10 % longer (1.05 against 0.96 us; where the slices lie matters)
    ClusterEnd& s_end = *reinterpret_cast<ClusterEnd*>(smem_raw + H.smem);
    int* s_sent = reinterpret_cast<int*>(&s_end + 1);
    const int N = S.N, T = S.T, s = 3 * N, tid = threadIdx.x, NT = blockDim.x;
    constexpr int NV = 1 << VR;
    const int lg = LG >= 0 ? LG : H.lg, lanes = lg - VR, tpp = 1 << lanes, q = tid & (tpp - 1), cs = H.cs, npad = H.npad;
    const unsigned rank = cs > 1 ? cluster_rank() : 0u;
    const int chain = blockIdx.x / cs;
    const int first_i = euler_first(N, cs, (int)rank), mine = euler_first(N, cs, (int)rank + 1) - first_i;
    const int i = first_i + (tid >> lanes);
    const bool active = (tid >> lanes) < mine;
    const LJK<R>& k = S.k;
    R* X = pos + S.off + (long long)chain * S.chain_len;
    const R* Z = noise ? noise + S.off + (long long)chain * S.chain_len : X;
    R* buf = reinterpret_cast<R*>(smem_raw);  // two slices, then (lists) the positions at the last build
    R* ref = buf + 6 * npad;
    uint16_t* nbr = reinterpret_cast<uint16_t*>(ref + (LIST ? 3 * npad : 0));
    EulerPos<R, LIST> P{buf, npad, lg};
    for (int j = tid; j < npad; j += NT)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            *P.at(j, c) = j < N ? X[c * N + j] : R(0);
            P.at(j, c)[3 * npad] = R(0);  // (padding of the other buffer)
        }
    int cnt[NV];  // list entries up to the end of each of this lane's sums (of four in the order
                  // in which they are added up: 0, 2, 1, 3)
    bool ovf = false;
    // candidates of this lane, sum by sum
    auto build = [&](const EulerPos<R, LIST>& A) {
        for (int j = tid; j < N; j += NT)
#pragma unroll
            for (int c = 0; c < 3; ++c) ref[c * npad + j] = *A.at(j, c);
        int n = 0;
        const R xi = active ? *A.at(i, 0) : R(0), yi = active ? *A.at(i, 1) : R(0), zi = active ? *A.at(i, 2) : R(0);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int sum = NV == 4 ? (v & 1) * 2 + (v >> 1) : v;
            for (int j = active ? q + sum * tpp : N; j < N; j += 1 << lg) {
                R dx, dy, dz;
                const R r2 = pair_r2<R>(xi, yi, zi, *A.at(j, 0), *A.at(j, 1), *A.at(j, 2), k, dx, dy, dz);
                if (r2 <= k.rl2 && j != i) {
                    if (n < H.cap && PAMD_OK_IDX(n * NT + tid, H.cap * NT)) nbr[n * NT + tid] = (uint16_t)j;
                    ++n;
                }
            }
            cnt[v] = n;
        }
        ovf = n > H.cap;
    };
    constexpr int NC = 3;
    const EulerLane lane(q, tpp, active);
    const int comp = lane.comp, first = lane.first, stride = lane.stride, nc = lane.nc;
    const bool mover = lane.mover, owner = lane.owner;
    const int oi = (int)(P.at(active ? i : 0, 0) - buf);
    R* const W = buf + oi + comp * npad;                       // own component, buffer 0
    const R* zp = Z + (long long)s + comp * N + (active ? i : 0);  // its normal of the step to load next
    R* xp = X + (long long)comp * N + (active ? i : 0);            // its place in slice t
    // (indexed by the unrolled step: copying a register would wait for its load)
    R z[2][NC], last[NC] = {R(0), R(0), R(0)};
    auto load_zs = [&](bool in, R (&v)[NC]) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < nc) v[c] = (in && mover) ? zp[c * N] : R(0);
        zp += s;
    };
    load_zs(true, z[0]);
    load_zs(T > 1, z[1]);
    // Slice t + 1 goes to the buffer that slice t - 1 was in.  A particle's slice t + 1 is sent
    // after every slice t has arrived, so after every CTA is done with slice t - 1 (its own
    // particles' slice t followed from it); the last lanes to read it are those that send.
    // A barrier is armed for slice t + 2 when slice t has arrived on it.  All of this needs a
    // particle in every CTA (euler_first): nothing would order the others behind one without.
    const unsigned bar0 = shared_addr(s_bar), bytes = (unsigned)(3 * N * sizeof(R));
    // A warp without particles does not wait, or it could fall two phases behind (with lists
    // the displacement check keeps all warps together).
    const bool waits = LIST || __any_sync(0xffffffffu, active);
    bool lost = false;  // a wait ran out: nothing is sent or armed any more, the steps count for nothing
    const int steps = (rank & 1u) ? min(T, max(1, limit.rounds)) : T;
    s_sent[tid] = steps;  // slices 1..steps are sent
    if (cs > 1)
        for (int j = tid; j < (int)(sizeof(ClusterEnd) / sizeof(unsigned)); j += NT) reinterpret_cast<unsigned*>(&s_end)[j] = 0u;
    if (cs > 1 && tid == 0) {
        barrier_init(bar0);
        barrier_init(bar0 + 8);
        barrier_init_done();
        expect(bar0 + 8, bytes);             // slice 1
        if (T > 1) expect(bar0, bytes);      // slice 2
    }
    if (cs > 1)
        cluster_barrier();
    else
        __syncthreads();
    // (also: every lane holds its first normals before slice 1 is written)
    const DenseForce<LG >= 0 ? LG : 0> dense(dense_consts(k), N, npad, i);
    // Step t from buffer PAR to the other; zt: its normals, then those of step t + 2.  The slice that the step before
    // made is stored here: a store directly before the barrier would hold it up (the
    // barrier's release waits for it).
    auto step = [&](int t, auto par, R (&zt)[NC]) {
        constexpr int PAR = decltype(par)::value;
        const EulerPos<R, LIST> A{buf + PAR * 3 * npad, npad, lg};
        if (t > 0 && owner) {
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (c < nc) xp[c * N] = last[c];
        }
        xp += s;
        if (cs > 1 && tid == 0 && t > 0 && t + 2 <= T && !lost) expect(bar0 + 8 * PAR, bytes);
        if (LIST) {
            bool moved = t == 0;
            for (int j = tid; j < N; j += NT) {
                const R dx = *A.at(j, 0) - ref[j], dy = *A.at(j, 1) - ref[npad + j], dz = *A.at(j, 2) - ref[2 * npad + j];
                moved |= !(dx * dx + dy * dy + dz * dz <= k.hs2);
            }
            if (__syncthreads_or(moved)) {
                build(A);
                __syncthreads();
            }
        }
        R f[3] = {R(0), R(0), R(0)}, xi[3] = {R(0), R(0), R(0)};
        if (active) {
#pragma unroll
            for (int c = 0; c < 3; ++c) xi[c] = A.p[oi + c * npad];
            if (LIST && !ovf) {
                // one loop over the entries of all sums (a loop for each would take the longest
                // lane's entries in every one of them: up to 1.5 times as long in double)
                R g[3] = {R(0), R(0), R(0)}, g1[3] = {R(0), R(0), R(0)};
                auto turn = [&](int m) {  // entry m is the first of another sum
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        if (m == cnt[0]) g[c] = f[c], f[c] = R(0);
                        if (NV == 4 && m == cnt[1 % NV]) g[c] += f[c], f[c] = R(0);
                        if (NV == 4 && m == cnt[2 % NV]) g1[c] = f[c], f[c] = R(0);
                    }
                };
#pragma unroll 2
                for (int m = 0; m < cnt[NV - 1]; ++m) {
                    if (NV > 1) turn(m);
                    const int j = nbr[m * NT + tid];
                    pair_force<R>(xi[0], xi[1], xi[2], *A.at(j, 0), *A.at(j, 1), *A.at(j, 2), k, f);
                }
                if (NV > 1) {
                    turn(cnt[NV - 1]);
#pragma unroll
                    for (int c = 0; c < 3; ++c) f[c] = NV == 4 ? g[c] + (g1[c] + f[c]) : g[c] + f[c];
                }
            } else {
                sum_tree<R, 0, 1, NV>(f, [&](auto sum, R (&f)[3]) {
                    constexpr int v = decltype(sum)::value;
                    const int j0 = q + v * tpp, dj = 1 << lg;  // candidates j0, j0 + dj, ...
                    f[0] = f[1] = f[2] = R(0);
                    if constexpr (sizeof(R) == 8 && LG == kOrderedLg) {
                        for (int j = j0; j < N; j += dj)
                            if (j != i) {
                                R dx, dy, dz;
                                const R r2 = pair_r2<R>(xi[0], xi[1], xi[2], *A.at(j, 0), *A.at(j, 1), *A.at(j, 2), k, dx, dy, dz);
                                if (!(r2 <= k.rc2)) continue;
                                const R ri = rsqrt(r2), ir2 = ri * ri, ir6 = ir2 * ir2 * ir2, u = k.c1 * ir6;
                                const R fs = fma_r(u * fma_r(k.c2, ir6, R(-1)), ir2, k.duc * ri);
                                f[0] = fma_r(fs, dx, f[0]);
                                f[1] = fma_r(fs, dy, f[1]);
                                f[2] = fma_r(fs, dz, f[2]);
                            }
                    } else if constexpr (LG >= 0) {
                        dense.template sum<(VR > 0)>(A.p, xi, j0, f);
                    } else {
                        for (int j = j0; j < N; j += dj)
                            if (j != i) pair_force<R>(xi[0], xi[1], xi[2], *A.at(j, 0), *A.at(j, 1), *A.at(j, 2), k, f);
                    }
                });
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (o < tpp)
#pragma unroll
                for (int c = 0; c < 3; ++c) f[c] += __shfl_xor_sync(0xffffffffu, f[c], o);
        auto move = [&](int c, R x, R fc, R zc) {
            const R xn = x + fma_r(k.a, fc, k.sig_em * zc);
            last[c] = xn;
            R* w = W + (1 - PAR) * 3 * npad + c * npad;
            if (cs == 1) {
                if (owner) *w = xn;
            } else if (!lost) {
                const unsigned to = shared_addr(w), bar = bar0 + 8 * (1 - PAR);
                for (int d = first; d < cs; d += stride)
                    send_async(remote_addr(to, (unsigned)d), xn, remote_addr(bar, (unsigned)d));
            }
        };
        if (mover) {
            if (tpp >= 3) {
                move(0, comp == 0 ? xi[0] : comp == 1 ? xi[1] : xi[2], comp == 0 ? f[0] : comp == 1 ? f[1] : f[2], zt[0]);
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) move(c, xi[c], f[c], zt[c]);
            }
        }
        load_zs(t + 2 < T, zt);
        if (cs == 1)
            __syncthreads();
        else if (waits && !lost && !wait_phase(bar0 + 8 * (1 - PAR), (unsigned)(t >> 1) & 1u, limit))
            lost = true, s_sent[tid] = t + 1;
    };
    using P0 = std::integral_constant<int, 0>;
    using P1 = std::integral_constant<int, 1>;
    for (int t = 0; t < steps; t += 2) {
        step(t, P0{}, z[0]);
        if (t + 1 < steps) step(t + 1, P1{}, z[1]);
    }
    if (owner) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < nc) xp[c * N] = last[c];
    }
    if (cs > 1) {
        if (cluster_lost(&s_end, lost || steps < T, cs)) {
            euler_drain<R>(&s_end, s_sent, shared_addr(s_bar), S.N, S.T, H.cs, lanes, X);
            if (tid == 0) atomicExch(err, PAMD_ERR_TIMEOUT);
        }
    }
}

template <typename R>
using EulerKernel = void (*)(R*, const R*, LJSysDev<R>, EulerShape, int*, WaitLimit);
template <typename R, bool LIST, int LG>
EulerKernel<R> euler_kernel_vr(const EulerShape& h)
{
    if (h.nt <= 512)
        return h.vr == 0   ? lj_euler_kernel<R, LIST, LG, 0, 512>
               : h.vr == 1 ? lj_euler_kernel<R, LIST, LG, 1, 512>
                           : lj_euler_kernel<R, LIST, LG, 2, 512>;
    return h.vr == 0   ? lj_euler_kernel<R, LIST, LG, 0, 1024>
           : h.vr == 1 ? lj_euler_kernel<R, LIST, LG, 1, 1024>
                       : lj_euler_kernel<R, LIST, LG, 2, 1024>;
}
template <typename R>
EulerKernel<R> euler_kernel(int N, const EulerShape& h)
{
    if (N > kEulerDense) return euler_kernel_vr<R, true, -1>(h);
    if (h.lg == kOrderedLg) return lj_euler_kernel<R, false, kOrderedLg, 0, 512>;  // (N <= kEulerOrdered)
    if constexpr (sizeof(R) == 8)
        return euler_kernel_vr<R, false, -1>(h);
    else
        return h.lg == 5 ? euler_kernel_vr<R, false, 5>(h) : h.lg == 4 ? euler_kernel_vr<R, false, 4>(h) : nullptr;
}

}  // namespace

template <typename R>
cudaError_t launch_lj_euler(R* pos, const R* noise, const void* sys_entry_host, int n_chains, int chain0,
                            uint64_t seed, uint64_t counter, int* err, const WaitLimit& limit, cudaStream_t st)
{
    const LJSysDev<R> S = *static_cast<const LJSysDev<R>*>(sys_entry_host);
    if (n_chains <= 0 || S.T <= 0) return cudaSuccess;
    int dev = 0, sms = 0, max_smem = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if (!noise) {
        const long long ng = S.chain_len / 4 + 1;
        const dim3 grid((unsigned)n_chains, (unsigned)std::min<long long>(1024, (ng + 255) / 256));
        euler_normals_kernel<R><<<grid, 256, 0, st>>>(pos, S.off, S.chain_len, 3 * S.N, chain0, seed, counter);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const double rl2 = (double)S.k.rl2, L = (double)S.k.L;
    const EulerShape h = euler_shape<R>(S.N, n_chains, 4.18879020478639 * rl2 * std::sqrt(rl2) * S.N / (L * L * L), sms,
                                        max_smem - 6 * 1024);
    const EulerKernel<R> kern = euler_kernel<R>(S.N, h);
    if (!kern) return cudaErrorInvalidValue;
    const size_t smem = h.smem + sizeof(ClusterEnd) + sizeof(int) * (size_t)h.nt;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_chains * h.cs));
    cfg.blockDim = dim3((unsigned)h.nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)h.cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = h.cs > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, pos, noise, S, h, err, limit);
}

template cudaError_t launch_lj_euler<float>(float*, const float*, const void*, int, int, uint64_t, uint64_t, int*,
                                            const WaitLimit&, cudaStream_t);
template cudaError_t launch_lj_euler<double>(double*, const double*, const void*, int, int, uint64_t, uint64_t, int*,
                                             const WaitLimit&, cudaStream_t);

PAMD_DEBUG_FETCHER(lj_euler)

}  // namespace pamd
