// dfloat.cuh -- pairs of FP32 numbers (hi + lo, |lo| <= ulp(hi) / 2) for the FP64 passes over FP32 lattices.
//
// The equilibrium of the initial fields and the moments read back are computed in 64 bits and then rounded
// to, or summed from, FP32 values.  GB300's FP64 pipe does 2 operations a clock and SM, conversions
// included, 1/64 of the FP32 rate, so these passes over HBM-resident fields were bound by it: 2D Euler 8192^2,
// init 10.0 ms (now 1.42) and moments 6.0 ms against 0.95 ms of HBM each.  The pair operations below (error-free
// transformations of Dekker and Knuth with FMA) keep 45 bits or more at about ten FP32 instructions each.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "systems.cuh"

namespace eslbm {

struct dfloat {
    float hi, lo;
    dfloat() = default;
    __host__ __device__ constexpr dfloat(float h, float l) : hi(h), lo(l) {}
    // constants and host-side parameters; in device code only with constant arguments
    __host__ __device__ constexpr explicit dfloat(double v) : hi((float)v), lo((float)(v - (double)(float)v)) {}
    __host__ __device__ constexpr explicit dfloat(int v) : dfloat((double)v) {}
    __host__ __device__ constexpr explicit operator double() const { return (double)hi + (double)lo; }  // host side
};

// a + b = s + e exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// the same where |a| >= |b| (or a = 0)
__device__ __forceinline__ dfloat quick_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return dfloat(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ dfloat operator-(const dfloat &a) { return dfloat(-a.hi, -a.lo); }
__device__ __forceinline__ dfloat operator+(const dfloat &a, const dfloat &b)
{
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    return quick_sum(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ dfloat operator-(const dfloat &a, const dfloat &b) { return a + (-b); }
__device__ __forceinline__ dfloat operator*(const dfloat &a, const dfloat &b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return quick_sum(p, e);
}
__device__ __forceinline__ dfloat operator/(const dfloat &a, const dfloat &b)
{
    // 1 / b to 46 bits: one Newton step from the FP32 reciprocal, its residual formed exactly
    const float r = __frcp_rn(b.hi);
    float d = __fmaf_rn(-b.hi, r, 1.0f);
    d = __fmaf_rn(-b.lo, r, d);
    return a * quick_sum(r, __fmul_rn(r, d));
}
template <> __host__ __device__ __forceinline__ dfloat add_rn<dfloat>(dfloat a, dfloat b)
{
#ifdef __CUDA_ARCH__
    return a + b;
#else
    return a;  // device code only
#endif
}
template <> __host__ __device__ __forceinline__ dfloat sub_rn<dfloat>(dfloat a, dfloat b)
{
#ifdef __CUDA_ARCH__
    return a - b;
#else
    return a;
#endif
}

// Magnitudes: an expression in this type is the sum of the magnitudes of its terms, which bounds the terms that
// cancel in the expression itself (and so, times 2^-44, the error of its value in pairs).
struct fmag {
    float v;
    fmag() = default;
    __host__ __device__ constexpr explicit fmag(float x) : v(x < 0.0f ? -x : x) {}
    __host__ __device__ constexpr explicit fmag(double x) : fmag((float)x) {}
    __host__ __device__ constexpr explicit fmag(int x) : fmag((float)x) {}
    __device__ __forceinline__ explicit fmag(const dfloat &x) : v(fabsf(x.hi)) {}
};
__device__ __forceinline__ fmag operator+(const fmag &a, const fmag &b) { return fmag(a.v + b.v); }
__device__ __forceinline__ fmag operator-(const fmag &a, const fmag &b) { return fmag(a.v + b.v); }
__device__ __forceinline__ fmag operator*(const fmag &a, const fmag &b) { return fmag(a.v * b.v); }
__device__ __forceinline__ fmag operator/(const fmag &a, const fmag &b) { return fmag(__fdividef(a.v, b.v)); }
template <> __host__ __device__ __forceinline__ fmag add_rn<fmag>(fmag a, fmag b)
{
#ifdef __CUDA_ARCH__
    return a + b;
#else
    return a;
#endif
}
template <> __host__ __device__ __forceinline__ fmag sub_rn<fmag>(fmag a, fmag b)
{
#ifdef __CUDA_ARCH__
    return a + b;
#else
    return a;
#endif
}
// the constants that the equilibria read
__device__ __forceinline__ ParamsR<fmag> magnitudes(const ParamsR<dfloat> &p)
{
    ParamsR<fmag> q;
    q.V = fmag(p.V);
    q.inv2V = fmag(p.inv2V);
    for (int j = 0; j < 2; ++j) {
        q.a[j] = fmag(p.a[j]);
        q.c[j] = fmag(p.c[j]);
    }
    q.g = fmag(p.g);
    q.gamma_m1 = fmag(p.gamma_m1);
    for (int i = 0; i < 4; ++i) {
        q.ubar[i] = fmag(p.ubar[i]);
        q.aux[i] = fmag(p.aux[i]);
    }
    return q;
}

// v as a pair, in integer arithmetic; false (v left to FP64) unless v is zero or between 2^-LOW and 2^40: with LOW = 40
// no product of three such numbers and no residual of one leaves FP32's range.  Deviations (LOW = 70) may be smaller:
// what their products lose is below the smallest FP32 number.
template <unsigned LOW = 40> __device__ __forceinline__ bool to_pair(double v, dfloat &p)
{
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
    const uint32_t mag = h & 0x7fffffffu, sign = h & 0x80000000u;
    const float top = __uint_as_float(sign | ((mag - (896u << 20)) << 3) | (l >> 29));  // towards zero
    const float unit = __uint_as_float(sign | (((mag >> 20) - 896u - 52u) << 23));      // last place of v
    const bool zero = (mag | l) == 0u;
    p = quick_sum(top, __fmul_rn((float)(l & 0x1fffffffu), unit));
    if (zero) p = dfloat(0.0f, 0.0f);
    return zero || (mag >= ((1023u - LOW) << 20) && mag < ((1023u + 40u) << 20));
}

// out of line: inlined, its FP64 operations are issued ahead of the branch for every cell
static __device__ __noinline__ double sum_fp64(float a, float b, float c, float d)
{
    return (double)a + (double)b + (double)c + (double)d;
}

// The sum of Q floats as a double (to 2^-70 of the largest before that rounding): error-free sums in FP32, then
// three conversions and two additions in FP64 where summing in FP64 takes Q conversions and Q additions (16.8 M
// sums of four: 163 against 262 us).
// Sums that leave FP32 (overflow, infinities, NaN) are taken in FP64.
template <int Q> __device__ __forceinline__ double sum_exact(const float *f)
{
    float s, e;
    double r;
    if constexpr (Q == 2) {
        two_sum(f[0], f[1], s, e);
        r = (double)s + (double)e;
    } else {
        float s1, e1, s2, e2, e3, t, r1, u, r2;
        two_sum(f[0], f[1], s1, e1);
        two_sum(f[2], f[3], s2, e2);
        two_sum(s1, s2, s, e3);
        two_sum(e1, e2, t, r1);
        two_sum(t, e3, u, r2);
        r = (double)s + ((double)u + (double)__fadd_rn(r1, r2));
    }
    if (!(fabsf(s) <= 3.0e38f)) r = Q == 2 ? sum_fp64(f[0], f[1], 0.0f, 0.0f) : sum_fp64(f[0], f[1], f[Q - 2], f[Q - 1]);
    return r;
}

}  // namespace eslbm
