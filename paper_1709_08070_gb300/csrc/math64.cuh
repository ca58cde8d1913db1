// FP64 helpers for kernels bound by the FP64 pipe: reciprocal and reciprocal
// square root for normal positive arguments without the special cases of the
// library functions, and integer forms of comparisons.
#pragma once
#include "ptx.cuh"

namespace ibim {

// 1/d and 1/sqrt(d) for normal positive d: the hardware estimate (about 20
// bits) and one third-order Newton (Halley) step, 1/d = y (1 + e + e^2 + ...)
// with e = 1 - d y, and 1/sqrt(d) = y (1 + e/2 + 3 e^2/8 + ...) with
// e = 1 - d y^2; the terms left out are below 2^-58.
__device__ __forceinline__ double rcp64(double d)
{
    const double y = ptx::rcp_approx64(d);
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

__device__ __forceinline__ double rsqrt64(double d)
{
    const double y = ptx::rsqrt_approx64(d);
    const double e = fma(-d * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// max(|a|, |b|) of finite values by their bit patterns (integer pipe).
__device__ __forceinline__ double max_abs64(double a, double b)
{
    const long long m = 0x7fffffffffffffffll;
    const long long x = __double_as_longlong(a) & m, y = __double_as_longlong(b) & m;
    return __longlong_as_double(x > y ? x : y);
}

// e^-x for x >= 0 from a table tab[i] = 2^(i/kExpTab) (Tang, ACM TOMS 15, 1989):
// x = -(k ln2/512 + u), |u| <= ln2/1024, e^u by its Taylor series to u^4 (the
// next term is below 2^-59), 2^(k/512) from the table and the exponent field.
// x is held at 700 (e^-x < 1e-304 there).  Nine FP64 instructions.
constexpr int kExpTab = 512;

__device__ __forceinline__ double exp_neg64(double x, const double* __restrict__ tab)
{
    const double xc = __double2hiint(x) > 0x4085e000 ? 700.0 : x;
    // round(-x 512/ln2) sits in the low word of the sum with 1.5 2^52
    const double t = fma(xc, -738.6598609351493, 6755399441055744.0);
    const int k = __double2loint(t);
    const double kf = t - 6755399441055744.0;
    double u = fma(kf, -0.0013538030871131923, -xc);  // ln2/512 in two parts, the first of 32 bits
    u = fma(kf, 8.204912251330243e-14, u);
    const double p = fma(u * u, fma(u, fma(u, 1.0 / 24.0, 1.0 / 6.0), 0.5), u);
    const double T = tab[k & (kExpTab - 1)];
    const double s = __hiloint2double(__double2hiint(T) + (k >> 9) * 1048576, __double2loint(T));
    return fma(s, p, s);
}

}  // namespace ibim
