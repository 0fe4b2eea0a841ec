// lj_double.cu -- double-precision Lennard-Jones path action and adjoint.
//
// What bounds it.  GB300 issues FP64 at 1/64 of the FP32 rate (two FMAs per SM
// and clock), so time is the number of FP64 instructions; single-precision and
// integer work, list traffic and memory are nearly free beside it.  The kernel
// therefore moves everything that does not have to be double off that pipe and
// evaluates the coefficients of a pair once:
//   * candidates, image shifts and the seed of 1/r come from single-precision
//     copies of the wrapped positions.  The neighbour test uses a radius widened by
//     more than its rounding error, so it admits every pair within the cutoff; the
//     decision r^2 <= rc^2 is then taken in double.
//   * an unordered pair i < j is evaluated once per slice (24 FP64 instructions):
//     pair vector, fs = -U'(r)/r and -(U'' - U'/r)/r^2, kept in a scratch of this
//     CTA in global memory.  The evaluation runs over a dense list of pairs, so no
//     lane idles.  (The scratch of all CTAs, 190 MB touched at N = 256, is more than
//     L2 holds: 587 MB read and 395 MB written in 0.95 ms, hidden behind the FP64 pipe.)
//   * force and Hessian-vector sums of particle i gather those records (3 and 13
//     FP64 instructions per neighbour), in increasing j.
// About 1600 FP64 instructions per particle-step at reduced density 0.85 and
// rc = 2.5, against about 7800 for the former form (Verlet lists of radius rc + 0.3,
// each ordered pair evaluated in the force and again in the Hessian-vector pass).
// Action and gradient of 2 x 512 steps of N = 256: 17.24 ms before (32 items of 32
// steps on 152 SMs, FP64 pipe 86 % busy on those), 0.95 ms now; the FP64 work alone
// takes 0.7 ms at 1.25 TFLOP/s.
//
// Formulas: the file lj_paired.cu states them; with ir2 = 1/r^2,
//   fs  = ir8 (c12 ir6 - c1) + u'(rc)/r,   nb = [ir8 (8 c1 - c23 ir6) - u'(rc)/r] ir2
//   (H v)_i = sum_j [fs w + nb (d . w) d],  w = v_j - v_i,  d = x_i - x_j.
// 1/r: inv_sqrt of lj_math.cuh (five FP64 instructions).
//
// Slices are independent up to r_{t-1} of the same particle, so a work item is a
// short run of slices of one chain (an atomic queue feeds a persistent grid); the
// first slice of an item leaves r_t and H r_t in `edge`, and lj_double_edge_kernel
// adds the residual of the step before it.  A result depends neither on the run
// length nor on the scratch capacity (a pair beyond the capacity is evaluated again
// where it is needed, by the same instructions).
#include <algorithm>
#include <type_traits>

#include "lj_math.cuh"

namespace pamd {

namespace {

// Threads and CTAs per SM, by what the shared memory of nmax particles allows: the FP64 pipe
// wants about 16 warps, of small systems more (their rows leave lanes idle); with two or fewer
// CTAs 128 registers are faster than 64.  Measured per particle-step: N = 256 4.15 ns with
// (256, 2), 3.6 with (256, 4); N = 500 4.8 with (256, 2), 6.0 with 64 registers; N = 864 9.9
// with one CTA of 256 threads, 7.2 with one of 512.
enum { kDblSmall = 0, kDblMedium = 1, kDblLarge = 2 };  // (256, 4), (256, 2), (512, 1)

// One pair's record: vector x_i - x_j (i < j) and fs; nb is kept beside it.
struct __align__(32) PairRec {
    double dx, dy, dz, fs;
};

// Scratch of one CTA: `cap` records, their nb and their particle indices, and the
// row prefixes when shared memory cannot hold them.
struct DblScratch {
    size_t rec, nb, ij, pre, bytes;
    __host__ __device__ DblScratch(int cap, int nmax, bool pre_global)
    {
        auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
        rec = 0;
        nb = rec + up(sizeof(PairRec) * (size_t)cap);
        ij = nb + up(sizeof(double) * (size_t)cap);
        pre = ij + up(sizeof(uint32_t) * (size_t)cap);
        bytes = pre + (pre_global ? up(sizeof(uint16_t) * (size_t)nmax * ((nmax + 31) / 32)) : 0);
    }
};

// Shared memory for nmax particles: positions and residuals (double), wrapped
// single-precision positions, box indices, slot bases, adjacency bits, prefixes.
struct DblSmem {
    size_t x, r, w, k, base, bits, pre, bytes;
    __host__ __device__ DblSmem(int nmax, bool pre_global)
    {
        const size_t n = (size_t)nmax, nw = (n + 31) / 32;
        auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
        w = 0;
        x = w + 16 * n;
        r = x + up(24 * n);
        k = r + up(24 * n);
        base = k + up(12 * n);
        bits = base + up(4 * n);
        pre = bits + up(4 * n * nw);
        bytes = pre + (pre_global ? 0 : up(2 * n * nw));
    }
};

// Exact double of a small integer (any integer, but those by the conversion instruction).
__device__ __forceinline__ double widen_int(int k)
{
    if (k > -(1 << 24) && k < (1 << 24)) return k == 0 ? 0.0 : widen((float)k);
    return (double)k;
}

// Everything the device functions need of one item's system.
struct DblCtx {
    int N, NW;
    LJK<double> k;
    float Lf, iLf, lim2, hbf;  // single-precision box, widened squared cutoff, image guard (negative: far slice)
    float4* W;
    double *X, *R;
    int *K, *base;
    uint32_t* bits;
    uint16_t* pre;
    PairRec* rec;
    double* nb;
    uint32_t* ij;
    int cap;

    __device__ __forceinline__ float image(float d) const
    {
        return __fsub_rn(__fmaf_rn(d, iLf, 12582912.0f), 12582912.0f);
    }
    // d = x_i - x_j, minimum image by the rule d = fma(-L, round(d (1/L)), d); fs and nb
    // (exact zeros outside the cutoff); r2 for the hard-sphere test.
    __device__ __forceinline__ void pair(int i, int j, PairRec& p, double& nbv, double& r2) const
    {
        const float4 a = W[i], b = W[j];
        const float fx = a.x - b.x, fy = a.y - b.y, fz = a.z - b.z;
        const float kx = image(fx), ky = image(fy), kz = image(fz);
        p.dx = X[3 * i] - X[3 * j];
        p.dy = X[3 * i + 1] - X[3 * j + 1];
        p.dz = X[3 * i + 2] - X[3 * j + 2];
        const float gx = fmaf(-Lf, kx, fx), gy = fmaf(-Lf, ky, fy), gz = fmaf(-Lf, kz, fz);
        double qx, qy, qz;
        if (fmaxf(fabsf(gx), fmaxf(fabsf(gy), fabsf(gz))) < hbf) {
            // away from half a box: the single-precision image is the nearest one
            qx = widen_int((int)kx + K[3 * i] - K[3 * j]);
            qy = widen_int((int)ky + K[3 * i + 1] - K[3 * j + 1]);
            qz = widen_int((int)kz + K[3 * i + 2] - K[3 * j + 2]);
        } else {
            const double m = 6755399441055744.0;  // 1.5 2^52: adding it rounds to an integer
            qx = __dsub_rn(__fma_rn(p.dx, k.iL, m), m);
            qy = __dsub_rn(__fma_rn(p.dy, k.iL, m), m);
            qz = __dsub_rn(__fma_rn(p.dz, k.iL, m), m);
        }
        p.dx = fma(-k.L, qx, p.dx);
        p.dy = fma(-k.L, qy, p.dy);
        p.dz = fma(-k.L, qz, p.dz);
        r2 = fma(p.dz, p.dz, fma(p.dy, p.dy, p.dx * p.dx));
        p.fs = 0.0;
        nbv = 0.0;
        // non-negative doubles compare as their bit patterns (a NaN compares above)
        if (__double_as_longlong(r2) <= __double_as_longlong(k.rc2)) {
            const double ri = inv_sqrt(r2), ir2 = ri * ri, ir6 = ir2 * ir2 * ir2, ir8 = ir6 * ir2;
            const double t = k.duc * ri;
            p.fs = fma(ir8, fma(k.c12, ir6, k.nc1), t);
            nbv = fma(ir8, fma(k.nc23, ir6, k.c8), -t) * ir2;
        }
    }
    // The record of the pair (i, j), from the lower index's side; evaluated again when
    // its slot lies beyond the capacity.
    template <bool NB>
    __device__ __forceinline__ PairRec record(int i, int j, int slot, double& nbv) const
    {
        PairRec p;
        if (slot < cap) {
            const double2* r = reinterpret_cast<const double2*>(rec + slot);
            const double2 a = r[0], b = r[1];
            p.dx = a.x;
            p.dy = a.y;
            p.dz = b.x;
            p.fs = b.y;
            if (NB) nbv = nb[slot];
        } else {
            double r2;
            pair(min(i, j), max(i, j), p, nbv, r2);
        }
        return p;
    }
    // Calls f(j, record, nb) for the neighbours j of i selected by `lanes` (bits j mod 32),
    // in increasing j; the records of four neighbours are loaded before the first is used.
    template <bool NB, typename F>
    __device__ __forceinline__ void neighbours(int i, uint32_t lanes, F&& f) const
    {
        const int wi = i >> 5;
        const uint32_t below_i = (1u << (i & 31)) - 1u;
        int w = -1, first = 0;
        uint32_t all = 0, m = 0;
        for (;;) {
            int js[4];
            PairRec p[4];
            double nbv[4];
            int n = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                while (m == 0 && ++w < NW) {
                    all = bits[i * NW + w];
                    m = all & lanes;
                    first = base[i] + pre[i * NW + w];
                }
                if (m != 0) {
                    const int b = __ffs(m) - 1;
                    const int j = 32 * w + b;
                    m &= m - 1;
                    const int slot = j > i ? first + __popc(all & ((1u << b) - 1u))
                                           : base[j] + pre[j * NW + wi] + __popc(bits[j * NW + wi] & below_i);
                    js[u] = j;
                    p[u] = record<NB>(i, j, slot, nbv[u]);
                    n = u + 1;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < n) f(js[u], p[u], nbv[u]);
            if (n < 4) break;
        }
    }
};

__device__ __forceinline__ double flip(double v, bool neg)
{
    return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000 : 0), __double2loint(v));
}

// HS: the hard-sphere path bias is on (hs2: squared radii, overlap: per global chain).
template <int NT, int MINB, bool GRAD, bool HS>
__global__ void __launch_bounds__(NT, MINB)
    lj_double_kernel(const LJItem* __restrict__ items, int n_items,
                     const LJSysDev<double>* __restrict__ systems, int nmax, int cap, int pre_global,
                     const double* __restrict__ pos, double* __restrict__ grad,
                     double* __restrict__ partials, int* __restrict__ counter,
                     unsigned char* __restrict__ scratch, double* __restrict__ edge,
                     const double* __restrict__ hs2, int* __restrict__ overlap)
{
    extern __shared__ __align__(32) unsigned char smem_raw[];
    constexpr int NWARP = NT / 32;
    __shared__ double red[NWARP];
    __shared__ int s_item, s_warp[NWARP];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DblScratch sc(cap, nmax, pre_global != 0);
    const DblSmem sl(nmax, pre_global != 0);
    unsigned char* mine = scratch + (size_t)blockIdx.x * sc.bytes;
    DblCtx C;
    C.W = reinterpret_cast<float4*>(smem_raw + sl.w);
    C.X = reinterpret_cast<double*>(smem_raw + sl.x);
    C.R = reinterpret_cast<double*>(smem_raw + sl.r);
    C.K = reinterpret_cast<int*>(smem_raw + sl.k);
    C.base = reinterpret_cast<int*>(smem_raw + sl.base);
    C.bits = reinterpret_cast<uint32_t*>(smem_raw + sl.bits);
    C.pre = pre_global ? reinterpret_cast<uint16_t*>(mine + sc.pre)
                       : reinterpret_cast<uint16_t*>(smem_raw + sl.pre);
    C.rec = reinterpret_cast<PairRec*>(mine + sc.rec);
    C.nb = reinterpret_cast<double*>(mine + sc.nb);
    C.ij = reinterpret_cast<uint32_t*>(mine + sc.ij);
    C.cap = cap;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= n_items) break;
        const LJItem I = items[it];
        const LJSysDev<double>& S = systems[I.sys];
        const int N = S.N, T = S.T, s = 3 * N;
        if (!PAMD_OK_IDX(N - 1, nmax)) continue;
        C.N = N;
        C.NW = (N + 31) >> 5;
        C.k = S.k;
        C.Lf = (float)C.k.L;
        C.iLf = 1.0f / C.Lf;
        // single-precision pair vectors of wrapped positions (|w| <= L/2) are within
        // 5e-7 L per component: r^2 within 2e-6 rc L + 3e-7 rc^2, ten times less than this
        const float rcf = sqrtf((float)C.k.rc2);
        C.lim2 = rcf * rcf + 2e-5f * rcf * (rcf + C.Lf);
        int lg = 0;  // threads per particle of the gathers: a power of two up to 8
        while (lg < 3 && (N << (lg + 1)) <= NT) ++lg;
        const int q = tid & ((1 << lg) - 1), per = NT >> lg;
        const uint32_t lanes = (lg == 0 ? 0xFFFFFFFFu : lg == 1 ? 0x55555555u : lg == 2 ? 0x11111111u
                                                                                          : 0x01010101u) << q;
        const double* __restrict__ Xg = pos + S.off + (long long)I.chain * S.chain_len;
        double* __restrict__ G = GRAD ? grad + S.off + (long long)I.chain * S.chain_len : nullptr;
        double* Ed = GRAD ? edge + (long long)I.slot * 9 * nmax : nullptr;  // r, H r of t0; r of t1 - 1
        // a slab's first item starts at its halo step, which only supplies r_{t0-1}
        const int ts = (S.halo_lo && I.t0 == S.halo_lo) ? I.t0 - 1 : I.t0;
        double acc = 0.0;
        bool ov = false;
        for (int t = ts; t < I.t1; ++t) {
            const double* Xt = Xg + (long long)t * s;
            // positions: double as stored, wrapped to [-L/2, L/2] in single precision.  Box
            // indices are kept in 32 bits: a slice with one of 2^30 or more (an exploding path)
            // takes its candidates and images in double
            bool far = false;
            for (int e = tid; e < s; e += NT) {
                if (!PAMD_OK_IDX((long long)t * s + e, (long long)(T + 1) * s)) continue;
                const int c = e / N, n = e - c * N;
                const double x = __ldg(Xt + e);
                const double m = __fma_rn(x, C.k.iL, 6755399441055744.0);
                // m = 1.5 2^52 + k, k the box index: |k| < 2^30 told from the words of m
                const int k = __double2loint(m);
                far |= (__double2hiint(m) != 0x43380000 + (k >> 31)) | ((unsigned)k + 0x40000000u >= 0x80000000u);
                C.X[3 * n + c] = x;
                C.K[3 * n + c] = k;
                reinterpret_cast<float*>(C.W + n)[c] = (float)__fma_rn(-C.k.L, __dsub_rn(m, 6755399441055744.0), x);
            }
            C.hbf = __syncthreads_or(far) ? -1.0f : 0.4999f * C.Lf;
            // adjacency rows: a warp per particle, 32 candidates per step
            auto search = [&](auto far_c) {
                for (int i = warp; i < N; i += NWARP) {
                    const float4 wi = C.W[i];
                    int cnt = 0;
                    for (int w = 0; w < C.NW; ++w) {
                        const int j = 32 * w + lane;
                        bool in = false;
                        if (j < N && !decltype(far_c)::value) {
                            const float4 wj = C.W[j];
                            float dx = wi.x - wj.x, dy = wi.y - wj.y, dz = wi.z - wj.z;
                            dx = fmaf(-C.Lf, C.image(dx), dx);
                            dy = fmaf(-C.Lf, C.image(dy), dy);
                            dz = fmaf(-C.Lf, C.image(dz), dz);
                            in = fmaf(dz, dz, fmaf(dy, dy, dx * dx)) <= C.lim2 && j != i;
                        } else if (decltype(far_c)::value && j < N && j != i) {
                            double ex, ey, ez;
                            in = pair_r2<double>(C.X[3 * i], C.X[3 * i + 1], C.X[3 * i + 2], C.X[3 * j], C.X[3 * j + 1],
                                                 C.X[3 * j + 2], C.k, ex, ey, ez) <= C.k.rc2;
                        }
                        const uint32_t m = __ballot_sync(0xffffffffu, in);
                        if (lane == 0) {
                            C.bits[i * C.NW + w] = m;
                            C.pre[i * C.NW + w] = (uint16_t)cnt;
                        }
                        cnt += __popc(m);
                    }
                }
            };
            if (C.hbf < 0.0f)
                search(std::true_type{});
            else
                search(std::false_type{});
            __syncthreads();
            // pairs j > i are numbered row by row: pair (i, j) has slot
            // base[i] + (neighbours of i below j); base[i] = pairs of earlier rows - neighbours below i
            const int rows = (N + NT - 1) / NT;  // consecutive rows of a thread (at most 4)
            int low[4], up[4], sum = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = tid * rows + u;
                low[u] = up[u] = 0;
                if (u < rows && i < N) {
                    const int o = i * C.NW, wi = i >> 5, wl = C.NW - 1;
                    low[u] = C.pre[o + wi] + __popc(C.bits[o + wi] & ((1u << (i & 31)) - 1u));
                    up[u] = C.pre[o + wl] + __popc(C.bits[o + wl]) - low[u];
                    sum += up[u];
                }
            }
            int inc = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += v;
            }
            if (lane == 31) s_warp[warp] = inc;
            __syncthreads();
            int run = inc - sum, total = 0;
#pragma unroll
            for (int v = 0; v < NWARP; ++v) {
                if (v < warp) run += s_warp[v];
                total += s_warp[v];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = tid * rows + u;
                if (u < rows && i < N) {
                    C.base[i] = run - low[u];
                    run += up[u];
                }
            }
            const int np = min(total, cap);
            __syncthreads();
            // the dense list of pairs
            for (int i = warp; i < N; i += NWARP) {
                const int b0 = C.base[i];
                for (int w = i >> 5; w < C.NW; ++w) {
                    const uint32_t all = C.bits[i * C.NW + w];
                    const int j = 32 * w + lane;
                    const int slot = b0 + C.pre[i * C.NW + w] + __popc(all & ((1u << lane) - 1u));
                    if (((all >> lane) & 1u) && j > i && slot < cap && PAMD_OK_IDX(slot, cap))
                        C.ij[slot] = (uint32_t)i | ((uint32_t)j << 16);
                }
            }
            __syncthreads();
            const double h2 = HS ? hs2[S.hs_off + t] : 0.0;
            for (int p = tid; p < np; p += NT) {
                const uint32_t v = C.ij[p];
                PairRec r;
                double nbv, r2;
                C.pair((int)(v & 0xFFFFu), (int)(v >> 16), r, nbv, r2);
                if (HS) ov |= (r2 <= C.k.rc2) & (r2 <= h2);
                double2* o = reinterpret_cast<double2*>(C.rec + p);
                o[0] = make_double2(r.dx, r.dy);
                o[1] = make_double2(r.dz, r.fs);
                if (GRAD) C.nb[p] = nbv;
            }
            if (HS && total > cap) {  // pairs without a record: tested from their rows
                for (int i = tid; i < N; i += NT)
                    for (int j = i + 1; j < N; ++j)
                        if ((C.bits[i * C.NW + (j >> 5)] >> (j & 31)) & 1u) {
                            PairRec r;
                            double nbv, r2;
                            C.pair(i, j, r, nbv, r2);
                            ov |= (r2 <= C.k.rc2) & (r2 <= h2);
                        }
            }
            __syncthreads();
            // forces, residuals
            const bool pending = GRAD && t == I.t0 && ts == I.t0 && t > 0;  // r_{t-1} is another item's
            for (int i0 = 0; i0 < N; i0 += per) {
                const int i = i0 + (tid >> lg);
                double f[3] = {0.0, 0.0, 0.0};
                if (i < N)
                    C.template neighbours<false>(i, lanes, [&](int j, const PairRec& p, double) {
                        const double fs = flip(p.fs, j < i);
                        f[0] = fma(fs, p.dx, f[0]);
                        f[1] = fma(fs, p.dy, f[1]);
                        f[2] = fma(fs, p.dz, f[2]);
                    });
                for (int o = (1 << lg) >> 1; o > 0; o >>= 1)
#pragma unroll
                    for (int c = 0; c < 3; ++c) f[c] += __shfl_xor_sync(0xffffffffu, f[c], o);
                if (i < N && q == 0) {
                    double r[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const long long e = (long long)(t + 1) * s + c * N + i;
                        const double xn = PAMD_OK_IDX(e, (long long)(T + 1) * s) ? __ldg(Xg + e) : 0.0;
                        r[c] = fma(-C.k.a, f[c], xn - C.X[3 * i + c]);
                        if (GRAD && t >= I.t0 && !pending) {
                            // r_{t-1} - r_t, completed below (r_{-1} = 0)
                            const double rp = t == 0 ? 0.0 : C.R[3 * i + c];
                            if (PAMD_OK_IDX(e - s, (long long)(T + 1) * s)) G[e - s] = rp - r[c];
                        }
                        C.R[3 * i + c] = r[c];
                        if (GRAD && pending) Ed[3 * i + c] = r[c];
                        if (GRAD && t == I.t1 - 1) Ed[6 * nmax + 3 * i + c] = r[c];
                    }
                    if (t >= I.t0) acc += fma(r[2], r[2], fma(r[1], r[1], r[0] * r[0]));
                }
            }
            __syncthreads();
            if (GRAD && t >= I.t0) {
                for (int i0 = 0; i0 < N; i0 += per) {
                    const int i = i0 + (tid >> lg);
                    double h[3] = {0.0, 0.0, 0.0};
                    if (i < N) {
                        const double vx = C.R[3 * i], vy = C.R[3 * i + 1], vz = C.R[3 * i + 2];
                        C.template neighbours<true>(i, lanes, [&](int j, const PairRec& p, double nbv) {
                            const double wx = C.R[3 * j] - vx, wy = C.R[3 * j + 1] - vy, wz = C.R[3 * j + 2] - vz;
                            const double bd = nbv * fma(p.dz, wz, fma(p.dy, wy, p.dx * wx));
                            h[0] = fma(p.fs, wx, fma(bd, p.dx, h[0]));
                            h[1] = fma(p.fs, wy, fma(bd, p.dy, h[1]));
                            h[2] = fma(p.fs, wz, fma(bd, p.dz, h[2]));
                        });
                    }
                    for (int o = (1 << lg) >> 1; o > 0; o >>= 1)
#pragma unroll
                        for (int c = 0; c < 3; ++c) h[c] += __shfl_xor_sync(0xffffffffu, h[c], o);
                    if (i < N && q == 0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const long long e = (long long)t * s + c * N + i;
                            if (!PAMD_OK_IDX(e, (long long)(T + 1) * s)) continue;
                            if (pending)
                                Ed[3 * nmax + 3 * i + c] = h[c];
                            else
                                G[e] = fma(C.k.a, h[c], G[e]) * C.k.ginv;
                        }
                    }
                }
                if (t == T - 1 && S.write_nose)
                    for (int e = tid; e < s; e += NT) {
                        const int c = e / N, n = e - c * N;
                        if (PAMD_OK_IDX((long long)T * s + e, (long long)(T + 1) * s))
                            G[(long long)T * s + e] = C.R[3 * n + c] * C.k.ginv;
                    }
            }
            __syncthreads();  // the slice's arrays are replaced next
        }
        if (HS && __syncthreads_or(ov) && tid == 0) atomicOr(overlap + S.chain0 + I.chain, 1);
        const double tot = block_sum(acc, red);
        if (tid == 0) partials[I.slot] = tot;
    }
}

// Gradient of the first slice of every item whose predecessor is another item:
// g = [r_{t-1} - r_t + a H r_t] / (2 D dt) from the two items' edge records.
__global__ void lj_double_edge_kernel(const LJItem* __restrict__ items, int n_items,
                                      const LJSysDev<double>* __restrict__ systems, int nmax,
                                      double* __restrict__ grad, const double* __restrict__ edge)
{
    const LJItem I = items[blockIdx.x];
    const LJSysDev<double>& S = systems[I.sys];
    if (I.t0 == 0 || I.t0 == S.halo_lo) return;
    const int N = S.N, s = 3 * N;
    const double* E = edge + (long long)I.slot * 9 * nmax;
    const double* P = edge + (long long)(I.slot - 1) * 9 * nmax + 6 * nmax;
    double* G = grad + S.off + (long long)I.chain * S.chain_len + (long long)I.t0 * s;
    const double a = S.k.a, ginv = S.k.ginv;
    for (int e = threadIdx.x; e < s; e += blockDim.x) {
        const int c = e / N, n = e - c * N;
        if (!PAMD_OK_IDX((long long)I.t0 * s + e, S.chain_len)) continue;
        G[e] = fma(a, E[3 * nmax + 3 * n + c], P[3 * n + c] - E[3 * n + c]) * ginv;
    }
}

using DoubleKernel = void (*)(const LJItem*, int, const LJSysDev<double>*, int, int, int, const double*,
                              double*, double*, int*, unsigned char*, double*, const double*, int*);
template <int NT, int MINB>
DoubleKernel double_kernel_of(bool grad, bool hs)
{
    if (grad) return hs ? lj_double_kernel<NT, MINB, true, true> : lj_double_kernel<NT, MINB, true, false>;
    return hs ? lj_double_kernel<NT, MINB, false, true> : lj_double_kernel<NT, MINB, false, false>;
}
DoubleKernel double_kernel(int form, bool grad, bool hs)
{
    return form == kDblSmall    ? double_kernel_of<256, 4>(grad, hs)
           : form == kDblMedium ? double_kernel_of<256, 2>(grad, hs)
                                : double_kernel_of<512, 1>(grad, hs);
}

}  // namespace

LJDoubleShape lj_double_shape(int nmax, double pairs_expected, int max_smem)
{
    LJDoubleShape h;
    const long long all = (long long)nmax * (nmax - 1) / 2;
    h.cap = (int)std::min<long long>(all, (long long)(1.25 * pairs_expected) + 64);
    h.pre_global = DblSmem(nmax, false).bytes > (size_t)max_smem;
    h.smem = DblSmem(nmax, h.pre_global).bytes;
    h.scratch = DblScratch(h.cap, nmax, h.pre_global).bytes;
    h.edge_doubles = 9 * nmax;
    const size_t each = h.smem + 1536;  // with the static and the reserved part
    h.form = 4 * each <= (size_t)max_smem ? kDblSmall : 2 * each <= (size_t)max_smem ? kDblMedium : kDblLarge;
    h.threads = h.form == kDblLarge ? 512 : 256;
    return h;
}

int lj_double_blocks_per_sm(const LJDoubleShape& h, bool with_grad)
{
    auto kern = double_kernel(h.form, with_grad, false);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)h.smem) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, h.threads, h.smem) != cudaSuccess) return 0;
    return nb;
}

cudaError_t launch_lj_double(const LJItem* items, int n_items, const void* sys_table, int nmax,
                             const LJDoubleShape& h, const double* pos, double* grad, double* partials,
                             int* counter, int grid, bool with_grad, unsigned char* scratch, double* edge,
                             cudaStream_t st, const double* hs2, int* overlap)
{
    if (n_items <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    auto kern = double_kernel(h.form, with_grad, hs2 != nullptr);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)h.smem);
    if (e != cudaSuccess) return e;
    const auto* sys = static_cast<const LJSysDev<double>*>(sys_table);
    kern<<<grid, h.threads, h.smem, st>>>(items, n_items, sys, nmax, h.cap, (int)h.pre_global, pos, grad,
                                            partials, counter, scratch, edge, hs2, overlap);
    e = cudaGetLastError();
    if (e != cudaSuccess || !with_grad) return e;
    lj_double_edge_kernel<<<n_items, 128, 0, st>>>(items, n_items, sys, nmax, grad, edge);
    return cudaGetLastError();
}

PAMD_DEBUG_FETCHER(lj_double)

}  // namespace pamd
