// FP64 arithmetic of the scheme with as few FP64-pipe operations as the results allow.
//
// GB300 issues about two FP64 operations per clock per SM, a sixtyfourth of its FP32 and a
// thirtysecond of its integer rate; comparisons, min/max and conversions of doubles run on
// the same pipe.  The FP64 kernels are bound by that pipe (84% active, 10% of the issue
// slots), so here
//   - reciprocal and division start from the hardware's approximations (rcp.approx.ftz.f64,
//     rsqrt.approx.ftz.f64, off the FP64 pipe) and take one third-order step (Householder;
//     Markstein 2000, "IA-64 and Elementary Functions", for the division's exact remainder):
//     3 operations for a reciprocal, 6 for a division.  Against 113-bit arithmetic, 8 million random
//     operands: the reciprocal within 0.506 ulp (0.03% differ from IEEE's, by one unit), every
//     division IEEE's;
//   - the sound speed sqrt(a / r) is one reciprocal square root of a r, 8 operations, within
//     1.0 ulp, rms 0.328 (a rounded square root of a rounded quotient: 0.85, rms 0.326);
//   - comparisons and MinMod are integer operations on the bit patterns, with the same
//     results, also for zeros (a zero MinMod up to its sign), infinities and NaN.
// Operands out of the middle of the exponent range take the IEEE operations (one function
// each, not inlined).
#pragma once
#include <cuda_runtime.h>

namespace amr {

// 2^-500 <= |x| < 2^500, by the high word
__device__ __forceinline__ bool mid_exp(double x)
{
    return (unsigned(__double2hiint(x)) & 0x7FFFFFFFu) - ((1023u - 500u) << 20) < (1000u << 20);
}
// the same and x > 0
__device__ __forceinline__ bool mid_exp_pos(double x)
{
    return unsigned(__double2hiint(x)) - ((1023u - 500u) << 20) < (1000u << 20);
}
__device__ __forceinline__ bool is_zero(double x)
{
    return ((unsigned(__double2hiint(x)) & 0x7FFFFFFFu) | unsigned(__double2loint(x))) == 0u;
}

static __device__ __noinline__ double div_ieee(double a, double b) { return a / b; }
static __device__ __noinline__ double sqrt_quot_ieee(double a, double r) { return sqrt(a / r); }

// 1/b, |b| in the middle range: x0 (1 + e + e^2), e = 1 - b x0
__device__ __forceinline__ double rcp_mid(double b)
{
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(b));
    const double e = __fma_rn(-b, x, 1.0);
    return __fma_rn(x, __fma_rn(e, e, e), x);
}

__device__ __forceinline__ double recip(double b) { return mid_exp(b) ? rcp_mid(b) : div_ieee(1.0, b); }

// a/b: the quotient by the reciprocal, corrected by its exact remainder
__device__ __forceinline__ double divide(double a, double b)
{
    if (mid_exp(b) && (mid_exp(a) || is_zero(a))) {
        const double x = rcp_mid(b), q = __dmul_rn(a, x);
        return __fma_rn(__fma_rn(-b, q, a), x, q);
    }
    return div_ieee(a, b);
}

// sqrt(a/r) = a / sqrt(a r).  The seed y has 21 significant bits, so y^2 is exact; with
// e = 1 - a r y^2, 1/sqrt(a r) = y (1 + e/2 + 3 e^2/8 + ...), and a y enters unrounded.
__device__ __forceinline__ double sqrt_quot(double a, double r)
{
    if (mid_exp_pos(a) && mid_exp_pos(r)) {
        const double t = __dmul_rn(a, r);
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(t));
        const double e = __fma_rn(-t, __dmul_rn(y, y), 1.0);
        const double s = __dmul_rn(__fma_rn(e, 0.375, 0.5), e);
        return __fma_rn(a, y, __dmul_rn(a, __dmul_rn(y, s)));
    }
    return sqrt_quot_ieee(a, r);
}

// x >= 0 and x > 0 for the result of an arithmetic operation (a NaN is a quiet one)
__device__ __forceinline__ bool ge0(double x)
{
    return unsigned(__double2hiint(x)) <= 0x7FF00000u || (__double2hiint(x) == int(0x80000000u) && __double2loint(x) == 0);
}
__device__ __forceinline__ bool gt0(double x)
{
    return unsigned(__double2hiint(x)) <= 0x7FF00000u && (__double2hiint(x) | __double2loint(x)) != 0;
}

// a > f ? a : f for a positive finite floor f: a's bits lie in (bits(f), bits(+Inf)]
__device__ __forceinline__ double floor_at(double a, double f)
{
    const unsigned long long ia = (unsigned long long)__double_as_longlong(a), jf = (unsigned long long)__double_as_longlong(f);
    return ia - jf - 1ull < 0x7FF0000000000000ull - jf ? a : f;
}

// MinMod of two differences (results of subtractions): zero when their signs differ or both are NaN,
// else the one of smaller magnitude; the other one when one is NaN.  The median (0, a, b) of
// fmin / fmax, bit for bit up to the sign of a zero.
__device__ __forceinline__ double minmod64(double a, double b)
{
    const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
    const unsigned long long top = 0x7FFFFFFFFFFFFFFFull;
    const unsigned long long ma = (unsigned long long)ia & top, mb = (unsigned long long)ib & top;
    const long long r = ma < mb ? ia : ib;
    const bool opposite = int(unsigned(ia >> 32) ^ unsigned(ib >> 32)) < 0;
    const unsigned ha = unsigned(ma >> 32), hb = unsigned(mb >> 32);
    const bool none_nan = max(ha, hb) <= 0x7FF00000u, both_nan = min(ha, hb) > 0x7FF00000u;
    return (opposite && none_nan) || both_nan ? 0.0 : __longlong_as_double(r);
}

}  // namespace amr
