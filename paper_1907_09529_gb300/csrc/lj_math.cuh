// lj_math.cuh -- arithmetic of the Lennard-Jones pair terms shared by the LJ kernels:
// packed f32x2 operations, the minimum-image rule, 1/r, and the pair force.
#pragma once

#include "pamd_internal.cuh"

namespace pamd {

// ------------------------------------------------------------------ packed f32x2 arithmetic
__device__ __forceinline__ float2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 pk(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b with one rounding: b * (-1) + a is exact before rounding.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, pk(-1.0f), a); }

// ------------------------------------------------------------------ double without conversions
// Float of a positive double by truncation (relative error below 2^-23), and the
// exact double of a float, by bit moves: conversion instructions run on the FP64 side.
__device__ __forceinline__ float trunc_to_float(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    return __uint_as_float(__funnelshift_l(lo, hi, 3) - 0xC0000000u);
}
__device__ __forceinline__ double widen(float f)  // normal f
{
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)),
                            (int)(b << 29));
}

// 1/sqrt(v).  Single precision: the hardware approximation (relative error below 2^-22).
__device__ __forceinline__ float inv_sqrt(float v)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
// Double: a single-precision seed (relative error e0 < 2^-21) and one third-order
// Householder iteration for the inverse square root,
//   e = 1 - v y^2,  y <- y + y e (1/2 + 3/8 e)     (remaining error 5/16 e^3),
// five FP64 instructions.  Outside the range where the seed's exponent fits a float (no
// physical distance) the library function is called.
__device__ __forceinline__ double inv_sqrt(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v);
    if (hi - 0x39000000u >= 0x46000000u - 0x39000000u) return rsqrt(v);
    const double y = widen(inv_sqrt(trunc_to_float(v)));
    const double e = fma(-(v * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// ------------------------------------------------------------------ pair terms
// Round-to-nearest-even of the exact product a*b (|a*b| < 2^22), by adding and
// removing 1.5*2^23 (float) or 1.5*2^52 (double): one FMA and one add.
__device__ __forceinline__ float round_prod(float a, float b)
{
    return __fsub_rn(__fmaf_rn(a, b, 12582912.0f), 12582912.0f);
}
__device__ __forceinline__ double round_prod(double a, double b)
{
    return __dsub_rn(__fma_rn(a, b, 6755399441055744.0), 6755399441055744.0);
}

// Minimum-image pair vector and |r_ij|^2 by the documented rule:
//   dx = xi - xj;  dx = fma(-L, round(dx * (1/L)), dx);  r2 = fma(dz,dz,fma(dy,dy,dx*dx)).
template <typename R>
__device__ __forceinline__ R pair_r2(R xi, R yi, R zi, R xj, R yj, R zj, const LJK<R>& k, R& dx, R& dy, R& dz)
{
    dx = xi - xj;
    dy = yi - yj;
    dz = zi - zj;
    dx = fma_r(-k.L, round_prod(dx, k.iL), dx);
    dy = fma_r(-k.L, round_prod(dy, k.iL), dy);
    dz = fma_r(-k.L, round_prod(dz, k.iL), dz);
    return fma_r(dz, dz, fma_r(dy, dy, mul_r(dx, dx)));
}
template <typename R>
__device__ __forceinline__ R pair_r2(R xi, R yi, R zi, const vec4_t<R>& pj, const LJK<R>& k, R& dx,
                                     R& dy, R& dz)
{
    return pair_r2<R>(xi, yi, zi, pj.x, pj.y, pj.z, k, dx, dy, dz);
}

// Pair scalars from r^2 (inside the cutoff):
//   fs  = -U'(r)/r = ir2 * u * t + u'(rc)/r,  u = c1 ir6, t = c2 ir6 - 1
//   upp = U''(r)   = ir2 * u * (c3 ir6 - 7)
template <typename R>
__device__ __forceinline__ R pair_fs(R r2, const LJK<R>& k, R& ir2, R& u, R& ir6)
{
    const R ri = inv_sqrt(r2);
    ir2 = ri * ri;
    ir6 = ir2 * ir2 * ir2;
    u = k.c1 * ir6;
    const R t = fma_r(k.c2, ir6, R(-1));
    return fma_r(u * t, ir2, k.duc * ri);
}

// The force of j on i, added to f; nothing outside the cutoff.
template <typename R>
__device__ __forceinline__ void pair_force(R xi, R yi, R zi, R xj, R yj, R zj, const LJK<R>& k, R (&f)[3])
{
    R dx, dy, dz, ir2, u, ir6;
    const R r2 = pair_r2<R>(xi, yi, zi, xj, yj, zj, k, dx, dy, dz);
    if (sizeof(R) == 8 && !(r2 <= k.rc2)) return;
    R fs = pair_fs<R>(r2, k, ir2, u, ir6);
    fs = (r2 <= k.rc2) ? fs : R(0);
    f[0] = fma_r(fs, dx, f[0]);
    f[1] = fma_r(fs, dy, f[1]);
    f[2] = fma_r(fs, dz, f[2]);
}

}  // namespace pamd
