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

}  // namespace ibim
