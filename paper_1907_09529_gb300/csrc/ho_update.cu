// ho_update.cu -- whole-path Metropolis-adjusted updates of harmonic systems.
//
// The oscillator's residuals and gradient couple an element only to its time
// neighbours e - s and e + s, so one pass over a block of elements can draw the
// proposal, form the action and gradient of the proposal and all three sums of the
// accept test; the neighbours just outside the block (s on either side) are proposed
// again here.  Arithmetic and summation orders are those of the separate kernels
// (mala_propose_kernel, ho_vec_kernel / ho_action_kernel, mala_reverse_kernel), so the
// results are bitwise the same.
//
//   ho_trial_kernel + mala_sums_accept_kernel + ho_commit_kernel: single precision, any length.
//     Memory traffic per coordinate 8 B read + 4 B written, then 4 + 8 B for accepted
//     chains: the gradient of the proposal is never stored, the commit pass forms it
//     again from the proposal.  The separate kernels move 48 B.
//   ho_loop_kernel: chains of one element block (up to 4096 elements).  One CTA per chain
//     keeps the path and its gradient in shared memory for all updates of the call.
//
// One update of 64 paths of 2^20 steps in 3D: 1645 us in the separate kernels, 979 us here
// (trial about 660, commit 310).
//
// What bounds them: ho_trial_kernel the instruction issue of Philox and Box-Muller (the
// normals are most of its instructions), ho_commit_kernel memory; ho_loop_kernel the
// latency of one update's chain of proposal, residuals, block sums and accept test, and in
// double precision the FP64 pipe of one SM (14 instructions per element at 16 clocks a warp).
#include "cluster.cuh"
#include "elem.cuh"

namespace pamd {

namespace {

constexpr int kHoMaxS = 64;  // elements per slice up to which the neighbours are proposed again

// Shared memory of one trial over a block of n elements (s per slice), in bytes.
template <typename R>
struct HoTrialSmem {
    size_t xp, zs, red, bytes;
    __host__ __device__ HoTrialSmem(int n, int s)
    {
        auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
        xp = 0;                                          // proposal with its neighbours
        zs = xp + up(sizeof(R) * ((size_t)n + 2 * s + 12));
        red = zs + up(sizeof(float) * ((size_t)n + 2 * s + 16));  // normals, then gradients
        bytes = red + sizeof(double) * 3 * kElemThreads;
    }
};

__device__ __forceinline__ float normal_r(float, float z) { return z; }
__device__ __forceinline__ double normal_r(double, float z) { return to_double(z); }

// One trial of block B: the proposal x' (to `prop` unless null), and this thread's sums
//   sums[0] += |r'|^2,  sums[1] += |x' - x + h g|^2,  sums[2] += |x - x' + h g'|^2.
// S: elements per slice when single precision and at most 4 (sums[0] in the order of
// ho_vec_kernel), else 0 (the order of ho_action_kernel).  XP, zs: HoTrialSmem.  gp: the
// gradient of the proposal, stored when not null.  pos, grad and gp may be shared memory.
// Returns the index of element 0 of the chain in XP.
template <typename R, int S>
__device__ __forceinline__ int ho_trial(const ElemBlock& B, const R* __restrict__ pos, const R* __restrict__ grad,
                                        R* __restrict__ prop, R* __restrict__ gp, R* XP, float* zs, R h, R s2h, R ak, R ginv, uint64_t seed, uint64_t counter,
                                        R (&sums)[3])
{
    constexpr bool F32 = sizeof(R) == 4;
    const int s = S ? S : B.s, tid = threadIdx.x;
    const int lo = B.e0 - s, hi = min(B.e0 + B.n + s, B.chain_len);
    const long long base = B.chain_base;
    const int off = (int)((base + lo) & 3) - lo;  // element e sits at XP[e + off]: aligned as in pos
    const int g0 = max(lo, 0) >> 2, g1 = (hi + 3) >> 2;
    const int xcap = B.n + 2 * s + 12;
    (void)xcap;
    for (int g = g0 + tid; g < g1; g += kElemThreads)
        if (PAMD_OK_IDX(4 * (g - g0) + 3, B.n + 2 * s + 16))
            *reinterpret_cast<float4*>(zs + 4 * (g - g0)) =
                philox_normals4(seed, counter, kStreamMala, (uint32_t)B.chain, (uint32_t)g);
    __syncthreads();
    auto step = [&](int e, R x, R g, R z, R& d) -> R {
        if (e < s) return x;  // the fixed tail x_0
        const R xp = x + fma_r(-h, g, s2h * z);
        d = xp - x;
        const R f = fma_r(h, g, d);
        sums[1] = fma_r(f, f, sums[1]);
        return xp;
    };
    ElemOrder<R> O(B);
    constexpr int KV = F32 ? kElemChunk / 4 / kElemThreads : 1;
    constexpr int K1 = F32 ? 1 : kElemChunk / kElemThreads;
    float dv[KV][4];
    R d1[K1];
#pragma unroll
    for (int k = 0; k < KV; ++k) {
        if (!O.vec(k)) break;
        const int q = O.rel(k), e = B.e0 + q;
        if (!PAMD_OK_IDX(e + 3, B.chain_len) || !PAMD_OK_IDX(e + off + 3, xcap)) continue;
        const float4 x = *reinterpret_cast<const float4*>(pos + base + e);
        const float4 g = *reinterpret_cast<const float4*>(grad + base + e);
        const float4 z = unaligned4(zs, e - 4 * g0);
        R d[4] = {R(0), R(0), R(0), R(0)};
        float4 o;
        o.x = (float)step(e, (R)x.x, (R)g.x, (R)z.x, d[0]);
        o.y = (float)step(e + 1, (R)x.y, (R)g.y, (R)z.y, d[1]);
        o.z = (float)step(e + 2, (R)x.z, (R)g.z, (R)z.z, d[2]);
        o.w = (float)step(e + 3, (R)x.w, (R)g.w, (R)z.w, d[3]);
#pragma unroll
        for (int l = 0; l < 4; ++l) dv[k][l] = (float)d[l];
        *reinterpret_cast<float4*>(XP + e + off) = o;
        if (prop) *reinterpret_cast<float4*>(prop + base + e) = o;
    }
#pragma unroll
    for (int k = 0; k < K1; ++k) {
        if (!O.one(k)) break;
        const int e = B.e0 + O.rel1(k);
        if (!PAMD_OK_IDX(e, B.chain_len) || !PAMD_OK_IDX(e + off, xcap)) continue;
        d1[k] = R(0);
        const R xp = step(e, pos[base + e], grad[base + e], normal_r(R(0), zs[e - 4 * g0]), d1[k]);
        XP[e + off] = xp;
        if (prop) prop[base + e] = xp;
    }
    // neighbours on either side (zeros beyond the ends of the chain; not summed)
    for (int q = tid; q < 2 * s; q += kElemThreads) {
        const int e = q < s ? lo + q : B.e0 + B.n + q - s;
        R xp = R(0);
        if (e >= 0 && e < B.chain_len) {
            const R x = pos[base + e];
            xp = e < s ? x : x + fma_r(-h, grad[base + e], s2h * normal_r(R(0), zs[e - 4 * g0]));
        }
        if (PAMD_OK_IDX(e + off, xcap)) XP[e + off] = xp;
    }
    __syncthreads();
    const int rend = B.chain_len - s;
    // residuals and gradient of the proposal at element e from (x_{e-s}, x_e, x_{e+s})
    auto grad_at = [&](int e, R xm, R x0, R xp, R& r) -> R {
        const R rp = (e >= s) ? fma_r(ak, xm, x0 - xm) : R(0);
        r = (e < rend) ? fma_r(ak, x0, xp - x0) : R(0);
        return fma_r(ak, r, rp - r) * ginv;
    };
    auto reverse = [&](int e, R g, R d) {
        if (e < s) return;
        const R b = fma_r(h, g, -d);  // x - x' is exactly -(x' - x)
        sums[2] = fma_r(b, b, sums[2]);
    };
    if (S > 0) {
#pragma unroll
        for (int k = 0; k < KV; ++k) {
            if (!O.vec(k)) break;
            const int e0 = B.e0 + O.rel(k);
            const R* c = XP + e0 + off;
            if (!PAMD_OK_IDX(e0 + off - 4, xcap) || !PAMD_OK_IDX(e0 + off + 7, xcap)) continue;
            const float4 P = *reinterpret_cast<const float4*>(c - 4), C = *reinterpret_cast<const float4*>(c),
                         Nx = *reinterpret_cast<const float4*>(c + 4);
            const float xx[12] = {P.x, P.y, P.z, P.w, C.x, C.y, C.z, C.w, Nx.x, Nx.y, Nx.z, Nx.w};
            float out[4];
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                R r;
                const R g = grad_at(e0 + l, (R)xx[4 + l - S], (R)xx[4 + l], (R)xx[4 + l + S], r);
                sums[0] = fma_r(r, r, sums[0]);
                reverse(e0 + l, g, (R)dv[k][l]);
                out[l] = (float)g;
            }
            if (gp) *reinterpret_cast<float4*>(gp + base + e0) = make_float4(out[0], out[1], out[2], out[3]);
        }
        if (O.one(0)) {
            const int e = B.e0 + O.rel1(0);
            R r;
            const R g = grad_at(e, XP[e - s + off], XP[e + off], XP[e + s + off], r);
            sums[0] = fma_r(r, r, sums[0]);
            reverse(e, g, d1[0]);
            if (gp) gp[base + e] = g;
        }
    } else {
        float* gs = zs;  // gradients in single precision: the reverse sum has another order
#pragma unroll
        for (int k = 0; k < kElemChunk / kElemThreads; ++k) {
            const int q = tid + k * kElemThreads, e = B.e0 + q;
            if (q >= B.n) break;
            if (!PAMD_OK_IDX(e - s + off, xcap) || !PAMD_OK_IDX(e + s + off, xcap)) continue;
            R r;
            const R g = grad_at(e, XP[e - s + off], XP[e + off], XP[e + s + off], r);
            sums[0] = fma_r(r, r, sums[0]);
            if (F32)
                gs[q] = (float)g;
            else
                reverse(e, g, d1[F32 ? 0 : k]);
            if (gp) gp[base + e] = g;
        }
        if (F32) {
            __syncthreads();
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                if (!O.vec(k)) break;
                const int q = O.rel(k), e = B.e0 + q;
                const float4 g = unaligned4(gs, q);
                reverse(e, (R)g.x, (R)dv[k][0]);
                reverse(e + 1, (R)g.y, (R)dv[k][1]);
                reverse(e + 2, (R)g.z, (R)dv[k][2]);
                reverse(e + 3, (R)g.w, (R)dv[k][3]);
            }
            if (O.one(0)) reverse(B.e0 + O.rel1(0), (R)gs[O.rel1(0)], d1[0]);
        }
    }
    return off;
}

template <typename R, int S>
__global__ void __launch_bounds__(kElemThreads)
    ho_trial_kernel(const ElemBlock* __restrict__ blocks, const R* __restrict__ pos, const R* __restrict__ grad,
                    R* __restrict__ prop, double* __restrict__ part_S, double* __restrict__ part_qf,
                    double* __restrict__ part_qr, const MalaDev* __restrict__ md, int update_index, R a, R ginv,
                    int max_s)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const HoTrialSmem<R> L(kElemChunk, max_s);
    const ElemBlock B = blocks[blockIdx.x];
    R sums[3] = {R(0), R(0), R(0)};
    ho_trial<R, S>(B, pos, grad, prop, nullptr, reinterpret_cast<R*>(smem_raw + L.xp),
                   reinterpret_cast<float*>(smem_raw + L.zs), step_h(*md, R(0)), step_s2h(*md, R(0)), a * harmonic_k(B, R(0)), ginv, md->seed,
                   md->counter + (uint64_t)update_index, sums);
    double tot[3] = {to_double(sums[0]), to_double(sums[1]), to_double(sums[2])};
    block_sums_256<3>(tot, reinterpret_cast<double*>(smem_raw + L.red));
    if (threadIdx.x == 0) {
        part_S[blockIdx.x] = tot[0];
        part_qf[blockIdx.x] = tot[1];
        part_qr[blockIdx.x] = tot[2];
    }
}

// Accepted chains: path <- proposal, gradient of the proposal formed from it, S <- S'.
template <typename R, int S>
__global__ void __launch_bounds__(kElemThreads)
    ho_commit_kernel(const ElemBlock* __restrict__ blocks, R* __restrict__ pos, R* __restrict__ grad,
                     const R* __restrict__ prop, const int* __restrict__ accept_flag, double* __restrict__ Sv,
                     const double* __restrict__ S_prop, R a, R ginv)
{
    const ElemBlock B = blocks[blockIdx.x];
    if (!accept_flag[B.chain]) return;
    const int s = S ? S : B.s;
    const R ak = a * harmonic_k(B, R(0));
    const R* __restrict__ X = prop + B.chain_base;
    const int rend = B.chain_len - s;
    auto grad_at = [&](int e, R xm, R x0, R xp) -> R {
        const R rp = (e >= s) ? fma_r(ak, xm, x0 - xm) : R(0);
        const R r = (e < rend) ? fma_r(ak, x0, xp - x0) : R(0);
        return fma_r(ak, r, rp - r) * ginv;
    };
    auto scalar = [&](int e) {
        if (!PAMD_OK_IDX(e, B.chain_len)) return;
        const R x0 = __ldg(X + e), xm = e >= s ? __ldg(X + e - s) : R(0), xp = e < rend ? __ldg(X + e + s) : R(0);
        pos[B.chain_base + e] = x0;
        grad[B.chain_base + e] = grad_at(e, xm, x0, xp);
    };
    if (S > 0) {
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        ElemOrder<float> O(B);
#pragma unroll 2
        for (int k = 0; O.vec(k); ++k) {
            const int e = B.e0 + O.rel(k);
            if (!PAMD_OK_IDX(e + 3, B.chain_len)) continue;
            const float4* v = reinterpret_cast<const float4*>(X + e);
            const float4 C = __ldg(v);
            const float4 P = e > 0 ? __ldg(v - 1) : z4;  // (holds an element of this chain)
            const float4 Nx = e + 4 < B.chain_len ? __ldg(v + 1) : z4;
            const float xx[12] = {P.x, P.y, P.z, P.w, C.x, C.y, C.z, C.w, Nx.x, Nx.y, Nx.z, Nx.w};
            float out[4];
#pragma unroll
            for (int l = 0; l < 4; ++l)
                out[l] = (float)grad_at(e + l, (R)xx[4 + l - S], (R)xx[4 + l], (R)xx[4 + l + S]);
            *reinterpret_cast<float4*>(pos + B.chain_base + e) = C;
            *reinterpret_cast<float4*>(grad + B.chain_base + e) = make_float4(out[0], out[1], out[2], out[3]);
        }
        if (O.one(0)) scalar(B.e0 + O.rel1(0));
    } else {
#pragma unroll 4
        for (int q = threadIdx.x; q < B.n; q += kElemThreads) scalar(B.e0 + q);
    }
    if (B.e0 == 0 && threadIdx.x == 0) Sv[B.chain] = S_prop[B.chain];
}

// All updates of chains of one block each: path, gradient, proposal and its gradient live in
// shared memory, laid out with the chain's alignment in the buffer.
template <typename R, int S>
__global__ void __launch_bounds__(kElemThreads)
    ho_loop_kernel(const ElemBlock* __restrict__ blocks, R* __restrict__ pos, R* __restrict__ grad,
                   double* __restrict__ Sv, const MalaDev* __restrict__ md, int update0, int n_updates, R a, R ginv,
                   double S_scale, const double* __restrict__ log_u, int* __restrict__ n_accepted,
                   double* __restrict__ log_alpha, int* __restrict__ err, int max_n, int max_s)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_acc;
    const HoTrialSmem<R> L(max_n, max_s);
    const size_t arr = (sizeof(R) * ((size_t)max_n + 4) + 15) & ~(size_t)15;
    ElemBlock B = blocks[blockIdx.x];
    const MalaDev M = *md;
    R* X = reinterpret_cast<R*>(smem_raw + L.bytes);
    R* G = reinterpret_cast<R*>(smem_raw + L.bytes + arr);
    R* GP = reinterpret_cast<R*>(smem_raw + L.bytes + 2 * arr);
    R* XP = reinterpret_cast<R*>(smem_raw + L.xp);
    const long long gbase = B.chain_base;
    const int mis = (int)(gbase & 3);
    for (int e = threadIdx.x; e < B.n; e += kElemThreads)
        if (PAMD_OK_IDX(mis + e, max_n + 4)) {
            X[mis + e] = pos[gbase + e];
            G[mis + e] = grad[gbase + e];
        }
    B.chain_base = mis;
    const int c = B.chain;
    double S_cur = Sv[c];
    int n_acc = 0;
    __syncthreads();
    for (int u = update0; u < update0 + n_updates; ++u) {
        R sums[3] = {R(0), R(0), R(0)};
        const int off = ho_trial<R, S>(B, X, G, (R*)nullptr, GP, XP, reinterpret_cast<float*>(smem_raw + L.zs),
                                       step_h(M, R(0)), step_s2h(M, R(0)), a * harmonic_k(B, R(0)), ginv, M.seed, M.counter + (uint64_t)u, sums);
        double tot[3] = {to_double(sums[0]), to_double(sums[1]), to_double(sums[2])};
        block_sums_256<3>(tot, reinterpret_cast<double*>(smem_raw + L.red));
        if (threadIdx.x == 0) {
            if (!isfinite(tot[0])) flag_nonfinite(err);
            const double S_new = tot[0] * S_scale;
            const int acc = mala_decide(c, S_cur, S_new, tot[1], tot[2], log_u, M, u,
                                        u == update0 + n_updates - 1 ? log_alpha : nullptr);
            if (acc) S_cur = S_new;
            n_acc += acc;
            s_acc = acc;
        }
        __syncthreads();
        if (s_acc) {
            for (int e = threadIdx.x; e < B.n; e += kElemThreads) X[mis + e] = XP[e + off];
            R* t = G;
            G = GP;
            GP = t;
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < B.n; e += kElemThreads)
        if (PAMD_OK_IDX(mis + e, max_n + 4)) {
            pos[gbase + e] = X[mis + e];
            grad[gbase + e] = G[mis + e];
        }
    if (threadIdx.x == 0) {
        Sv[c] = S_cur;
        if (n_accepted) n_accepted[c] += n_acc;
    }
}

// ------------------------------------------------------------------ double precision, few chains
// All updates of double-precision chains of one block, a cluster of CS = 2, 4 or 8 CTAs per
// chain.  One SM issues the 14 FP64 instructions of an element at two lanes a clock, and the
// update is a chain of dependent steps, so the elements are spread over the cluster, one per
// thread.  The sums keep ho_loop_kernel's order: its thread v adds elements v, v + 256, ..., so
// CTA `rank` takes the runs [256 k + 32 VW rank, + 32 VW) of every k (VW = 8 / CS of the eight
// warps), forms their terms, adds them per v in increasing k and over each warp, and sends the
// warp sums to every CTA; each then takes the accept test itself.  The s elements on either
// side of a run are proposed again here; their gradients come from the CTA that owns them.
// One exchange per update, during which the next normals are drawn; log u of kLuBatch
// updates at a time, and the accept test without its two divisions where they cannot decide it.
// 100 updates of one path of 1024 steps: 918 us with ho_loop_kernel, 308 us here (360 us with
// log u per update, the divisions in every test, and a cluster barrier).  Of an update's 5900
// cycles about 700 go to the trial positions, 1300 to gradients and terms, 1650 to the warp sums
// (five dependent FP64 additions), 1100 to the exchange (the normals within it), 1500 to the
// eight-warp sums and the test: FP64 latency throughout.
constexpr int kLuBatch = 64;

struct HoCluster {
    int cs, vw, K, s;  // CTAs, warps of the sum order per CTA, runs per CTA, elements per slice
    __host__ __device__ int run() const { return 32 * vw; }
    __host__ __device__ int own() const { return 32 * vw * K; }
    __host__ __device__ int halo() const { return 2 * s * K; }
    __host__ __device__ int threads() const { return own() + (halo() + 31) / 32 * 32; }
    // whether the run before (after) has a copy of the gradient at place p of run k, and its CTA
    __device__ bool to_prev(unsigned rank, int k, int p) const { return p < s && (rank > 0 || k > 0); }
    __device__ bool to_next(unsigned rank, int k, int p) const { return p >= run() - s && ((int)rank < cs - 1 || k < K - 1); }
    __device__ unsigned prev(unsigned rank) const { return rank > 0 ? rank - 1 : cs - 1; }
    __device__ unsigned next(unsigned rank) const { return (int)rank < cs - 1 ? rank + 1 : 0u; }
    __host__ __device__ size_t doubles() const  // x', terms, halo gradients (2), warp sums (2)
    {
        return (size_t)K * (run() + 2 * s) + 3 * (size_t)own() + 2 * (size_t)halo() + 2 * 24;
    }
};

// After a lost wait of a cluster.  A thread has sent its part of `sent[tid]` updates; mine: its
// element is one of the CTA's, at place p of run k.
__device__ __noinline__ void ho_cluster_drain(ClusterEnd* E, const int* sent, const int* armed, unsigned bar0,
                                              unsigned bytes, bool mine, int k, int p, const HoCluster& H)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const unsigned rank = cluster_rank();
    auto count = [&] {
        for (int b = 0; b < 2; ++b) {
            const unsigned n8 = 8u * (unsigned)((sent[tid] + 1 - b) / 2);  // of even, odd updates
            if (mine && H.to_prev(rank, k, p)) atomicAdd(&E->out[H.prev(rank)][b], n8);
            if (mine && H.to_next(rank, k, p)) atomicAdd(&E->out[H.next(rank)][b], n8);
            for (int q = tid >> 5; q < 3 * H.vw; q += blockDim.x >> 5)
                if (lane < H.cs) atomicAdd(&E->out[lane][b], n8);
        }
    };
    cluster_drain(E, bar0, bytes, H.cs, [&](int b) { return (unsigned)((*armed + 1 - b) / 2); }, count);
}

__global__ void __launch_bounds__(1024)
    ho_cluster_kernel(const ElemBlock* __restrict__ blocks, double* __restrict__ pos, double* __restrict__ grad,
                      double* __restrict__ Sv, const MalaDev* __restrict__ md, int update0, int n_updates, double a,
                      double ginv, double S_scale, const double* __restrict__ log_u, int* __restrict__ n_accepted,
                      double* __restrict__ log_alpha, int* __restrict__ err, const HoCluster H, const WaitLimit limit)
{
    extern __shared__ __align__(16) double smem_d[];
    __shared__ int s_acc;
    __shared__ double s_lu[kLuBatch];
    __shared__ __align__(8) uint64_t s_bar[2];  // of even and odd updates
    __shared__ ClusterEnd s_end;
    __shared__ int s_sent[1024];  // updates a thread sends
    __shared__ int s_armed;
    __shared__ double s_la;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = blockDim.x >> 5;
    const int cs = H.cs, s = H.s, RL = H.run(), K = H.K, own_n = H.own(), pitch = RL + 2 * s;
    const unsigned rank = cluster_rank();
    const ElemBlock B = blocks[blockIdx.x / cs];
    const MalaDev M = *md;
    PAMD_ARR(double, XP, smem_d, K * pitch);
    PAMD_ARR(double, V, smem_d + K * pitch, 3 * own_n);
    double* HG = smem_d + K * pitch + 3 * own_n;  // [2][halo]
    double* VS = HG + 2 * H.halo();               // [2][3][8]
    // this thread's element: one of the CTA's runs, or a neighbour of one
    const bool own = tid < own_n;
    const int h = tid - own_n;
    const bool halo = h >= 0 && h < H.halo();
    const int k = own ? tid / RL : halo ? h / (2 * s) : 0;
    const int p = own ? tid - k * RL : halo ? ((h / s) & 1 ? RL + h % s : h % s - s) : 0;  // place in the run
    const int e = 256 * k + RL * (int)rank + p;
    const bool in = (own || halo) && e >= 0 && e < B.n;
    const bool moves = in && e >= s;  // not the fixed tail x_0
    const int xi = k * pitch + s + p;
    const double ak = a * B.k, hh = M.h, s2h = M.s2h;
    const int rend = B.chain_len - s;
    double* gx = pos + B.chain_base + e;
    double* gg = grad + B.chain_base + e;
    double x = in ? *gx : 0.0, g = in ? *gg : 0.0, S_cur = Sv[B.chain];
    int n_acc = 0;
    auto normal = [&](int u) -> double {
        if (!moves) return 0.0;
        const float4 q = philox_normals4(M.seed, M.counter + (uint64_t)u, kStreamMala, (uint32_t)B.chain, (uint32_t)(e >> 2));
        return to_double(pick4(q, e & 3));
    };
    // log u of updates u .. u + kLuBatch - 1, one per thread: a double logarithm takes longer
    // than the barrier's round trip
    auto draw_lu = [&](int u) {
        for (int q = tid; q < kLuBatch && u + q < update0 + n_updates; q += blockDim.x)
            s_lu[q] = log_u ? log_u[B.chain]
                            : log(philox_uniform53(M.seed, M.counter + (uint64_t)(u + q), kStreamAccept,
                                                   (uint32_t)B.chain));
    };
    const double h4 = 4.0 * hh, h4_inv = 1.0 / h4;
    double z = normal(update0);
    if (own || halo) XP[xi] = 0.0;
    for (int j = tid; j < (int)(sizeof(ClusterEnd) / sizeof(unsigned)); j += blockDim.x) reinterpret_cast<unsigned*>(&s_end)[j] = 0u;
    // Received per update: 24 warp sums and the gradients of this CTA's halo elements.  Those of
    // update n + 2 replace those of update n: they are sent after the sums of update n + 1 have
    // come from every CTA, so after every thread of every CTA is done with update n.
    const unsigned bar0 = shared_addr(s_bar), bytes = 8u * (24u + (unsigned)__syncthreads_count(halo && in));
    bool lost = false;
    const int rounds = (rank & 1u) ? min(n_updates, limit.rounds) : n_updates;
    s_sent[tid] = rounds;
    if (tid == 0) {
        barrier_init(bar0);
        barrier_init(bar0 + 8);
        barrier_init_done();
        expect(bar0, bytes);
        if (n_updates > 1) expect(bar0 + 8, bytes);
    }
    cluster_barrier();
    for (int u = update0; u < update0 + rounds; ++u) {
        const int n = u - update0, par = n & 1, lu_at = n % kLuBatch;
        const unsigned bar = bar0 + 8 * par;
        auto send = [&](double* p, unsigned to, double v) {
            send_async(remote_addr(shared_addr(p), to), v, remote_addr(bar, to));
        };
        if (lu_at == 0) draw_lu(u);
        const double xp = moves ? x + fma_r(-hh, g, s2h * z) : x;
        if (in) XP[xi] = xp;
        __syncthreads();
        double gp = 0.0;
        if (own) {
            double r = 0.0, f = 0.0, b = 0.0;
            if (in) {
                const double xm = XP[xi - s], xn = XP[xi + s];
                const double rp = e >= s ? fma_r(ak, xm, xp - xm) : 0.0;
                r = e < rend ? fma_r(ak, xp, xn - xp) : 0.0;
                gp = fma_r(ak, r, rp - r) * ginv;
                if (moves) {
                    const double d = xp - x;
                    f = fma_r(hh, g, d);
                    b = fma_r(hh, gp, -d);
                }
                if (H.to_prev(rank, k, p) && !lost)
                    send(HG + par * H.halo() + (rank > 0 ? k : k - 1) * 2 * s + s + p, H.prev(rank), gp);
                if (H.to_next(rank, k, p) && !lost)
                    send(HG + par * H.halo() + ((int)rank < cs - 1 ? k : k + 1) * 2 * s + p - (RL - s), H.next(rank), gp);
            }
            V[tid] = r;
            V[own_n + tid] = f;
            V[2 * own_n + tid] = b;
        }
        __syncthreads();
        for (int q = warp; q < 3 * H.vw; q += NW) {
            const int w = q % H.vw, t = q / H.vw;
            double acc = 0.0;
            for (int kk = 0; kk < K; ++kk) {
                const double v = V[t * own_n + kk * RL + 32 * w + lane];
                acc = fma_r(v, v, acc);
            }
            acc = warp_sum(acc);
            if (lane < cs && !lost) send(VS + 24 * par + 8 * t + (int)rank * H.vw + w, (unsigned)lane, acc);
        }
        if (n + 1 < n_updates) z = normal(u + 1);
        asm volatile("" : "+d"(z));  // (here, not after the wait)
        // (lost: nothing is sent or armed any more, and nothing will be committed)
        if (!lost && !phase_done(bar, (unsigned)(n >> 1) & 1u) && !wait_phase(bar, (unsigned)(n >> 1) & 1u, limit))
            lost = true, s_sent[tid] = n + 1;
        if (tid == 32 * (NW - 1) && n + 2 < n_updates && !lost) expect(bar, bytes);  // (not by the accept test's warp: 1.3 us an update)
        if (warp == 0) {
            // lanes 8 t + w: sum t of warp w
            double v = lane < 24 ? VS[24 * par + lane] : 0.0;
            v += __shfl_xor_sync(0xffffffffu, v, 4);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            const double S_new = v * S_scale;  // lane 0; the others below in lanes 8 and 16
            const double qf = __shfl_sync(0xffffffffu, v, 8), qr = __shfl_sync(0xffffffffu, v, 16);
            if (lane == 0) {
                if (rank == 0 && !isfinite(v)) flag_nonfinite(err);
                // log alpha with the reciprocal of 4 h: within a few ulp of its largest term, so
                // the comparison is that of the divided form unless the two sides are that close
                // (two double divisions are most of this step otherwise)
                const double lu = s_lu[lu_at], a1 = qr * h4_inv, a2 = qf * h4_inv, dS = S_cur - S_new;
                double la = dS - a1 + a2;
                const bool last = u == update0 + n_updates - 1;
                if ((last && log_alpha) || !(fabs(lu - la) > 1e-12 * (fabs(dS) + a1 + a2))) la = dS - qr / h4 + qf / h4;
                const int acc = lu < la ? 1 : 0;  // NaN log alpha never accepts
                if (last) s_la = la;
                if (acc) S_cur = S_new;
                n_acc += acc;
                s_acc = acc;
            }
        }
        __syncthreads();
        if (s_acc) {
            x = xp;
            g = own ? gp : halo ? HG[par * H.halo() + h] : g;
        }
    }
    // updates armed: the first two, and n + 2 when the sums of update n had come
    if (tid == 32 * (NW - 1)) s_armed = min(n_updates, s_sent[tid] + (lost ? 1 : 2));
    if (cluster_lost(&s_end, lost || rounds < n_updates, cs)) {
        ho_cluster_drain(&s_end, s_sent, &s_armed, bar0, bytes, own && in, k, p, H);
        if (tid == 0) atomicExch(err, PAMD_ERR_TIMEOUT);  // the chain stays as it was
        return;
    }
    if (own && in) {
        *gx = x;
        *gg = g;
    }
    if (rank == 0 && tid == 0) {
        Sv[B.chain] = S_cur;
        if (n_accepted) n_accepted[B.chain] += n_acc;
        if (log_alpha) log_alpha[B.chain] = s_la;
    }
}

// The cluster shape for chains of n elements, s to a slice: as many CTAs per chain (up to 8)
// as the GPU holds at once; cs = 0 where ho_loop_kernel is the better form (chains of less than
// kHoClusterMin elements, too many chains, wide slices).
constexpr int kHoClusterMin = 200;
HoCluster ho_cluster_shape(int n_chains, int n, int s, int sms)
{
    HoCluster h{0, 0, (n + 255) / 256, s};
    if (n < kHoClusterMin || s > 16) return h;
    for (int cs = 8; cs >= 2; cs /= 2) {
        h.cs = cs;
        h.vw = 8 / cs;
        if ((long long)cs * n_chains <= sms && h.threads() <= 1024) return h;
    }
    h.cs = 0;
    return h;
}

}  // namespace

bool ho_update_fusable(int s) { return s <= kHoMaxS; }

template <typename R>
cudaError_t launch_ho_trial(const ElemBlock* blocks, int n_blocks, int s, const R* pos, const R* grad,
                            R* prop, double* part_S, double* part_qf, double* part_qr, const MalaDev* md,
                            int update_index, double a, double ginv, cudaStream_t st)
{
    if (n_blocks <= 0) return cudaSuccess;
    const size_t smem = HoTrialSmem<R>(kElemChunk, s).bytes;
    auto k = ho_trial_kernel<R, 0>;
    if (sizeof(R) == 4 && s >= 1 && s <= 4) {
        if constexpr (sizeof(R) == 4)
            k = s == 1   ? ho_trial_kernel<R, 1>
                : s == 2 ? ho_trial_kernel<R, 2>
                : s == 3 ? ho_trial_kernel<R, 3>
                             : ho_trial_kernel<R, 4>;
    }
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<n_blocks, kElemThreads, smem, st>>>(blocks, pos, grad, prop, part_S, part_qf, part_qr, md, update_index,
                                            (R)a, (R)ginv, s);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_ho_commit(const ElemBlock* blocks, int n_blocks, int s, R* pos, R* grad, const R* prop,
                             const int* accept_flag, double* S, const double* S_prop, double a, double ginv,
                             cudaStream_t st)
{
    if (n_blocks <= 0) return cudaSuccess;
    auto k = ho_commit_kernel<R, 0>;
    if (sizeof(R) == 4 && s >= 1 && s <= 4) {
        if constexpr (sizeof(R) == 4)
            k = s == 1   ? ho_commit_kernel<R, 1>
                : s == 2 ? ho_commit_kernel<R, 2>
                : s == 3 ? ho_commit_kernel<R, 3>
                             : ho_commit_kernel<R, 4>;
    }
    k<<<n_blocks, kElemThreads, 0, st>>>(blocks, pos, grad, prop, accept_flag, S, S_prop, (R)a, (R)ginv);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_ho_loop(const ElemBlock* blocks, int n_chains, int s, int max_n, R* pos, R* grad,
                           double* S, const MalaDev* md, int update0, int n_updates, double a, double ginv,
                           double S_scale, const double* log_u, int* n_accepted, double* log_alpha, int* err,
                           const WaitLimit& limit, cudaStream_t st)
{
    if (n_chains <= 0 || n_updates <= 0) return cudaSuccess;
    if constexpr (sizeof(R) == 8) {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const HoCluster h = ho_cluster_shape(n_chains, max_n, s, sms);
        if (h.cs) {
            const size_t bytes = sizeof(double) * h.doubles();
            if (bytes > 48 * 1024) {
                e = cudaFuncSetAttribute(ho_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
                if (e != cudaSuccess) return e;
            }
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(n_chains * h.cs));
            cfg.blockDim = dim3((unsigned)h.threads());
            cfg.dynamicSmemBytes = bytes;
            cfg.stream = st;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)h.cs;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            return cudaLaunchKernelEx(&cfg, ho_cluster_kernel, blocks, pos, grad, S, md, update0, n_updates, a, ginv,
                                      S_scale, log_u, n_accepted, log_alpha, err, h, limit);
        }
    }
    const size_t arr = (sizeof(R) * ((size_t)max_n + 4) + 15) & ~(size_t)15;
    const size_t smem = HoTrialSmem<R>(max_n, s).bytes + 3 * arr;
    auto k = ho_loop_kernel<R, 0>;
    if (sizeof(R) == 4 && s >= 1 && s <= 4) {
        if constexpr (sizeof(R) == 4)
            k = s == 1   ? ho_loop_kernel<R, 1>
                : s == 2 ? ho_loop_kernel<R, 2>
                : s == 3 ? ho_loop_kernel<R, 3>
                             : ho_loop_kernel<R, 4>;
    }
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<n_chains, kElemThreads, smem, st>>>(blocks, pos, grad, S, md, update0, n_updates, (R)a, (R)ginv, S_scale,
                                            log_u, n_accepted, log_alpha, err, max_n, s);
    return cudaGetLastError();
}

template cudaError_t launch_ho_trial<float>(const ElemBlock*, int, int, const float*, const float*, float*, double*,
                                            double*, double*, const MalaDev*, int, double, double, cudaStream_t);
template cudaError_t launch_ho_commit<float>(const ElemBlock*, int, int, float*, float*, const float*, const int*,
                                             double*, const double*, double, double, cudaStream_t);
#define PAMD_INST(R)                                                                                             \
    template cudaError_t launch_ho_loop<R>(const ElemBlock*, int, int, int, R*, R*, double*, const MalaDev*, \
                                           int, int, double, double, double, const double*, int*, double*, int*, \
                                           const WaitLimit&, cudaStream_t);
PAMD_INST(float)
PAMD_INST(double)
#undef PAMD_INST

PAMD_DEBUG_FETCHER(ho_update)

}  // namespace pamd
