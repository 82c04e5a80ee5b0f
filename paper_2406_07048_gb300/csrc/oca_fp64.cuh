// FP64 operations for the chains of the LQ solves, where an FP64 instruction holds a
// scheduler for 64 cycles whatever its lanes do.
#pragma once

#include <cuda_runtime.h>

namespace oca {

// 1 / x by one step of the third-order hyperpower iteration, y <- y + y (e + e^2) with
// e = 1 - x y (M. Altman, Pacific J. Math. 10, 1960; its second-order form is Schulz's),
// from the hardware's approximation.  That one keeps the upper 32 bits of its operand and
// of its result, so |e| < 2^-19 and what the step leaves, e^3, is below 2^-57 of 1 / x:
// with the rounding of the last multiply-add at most 0.57 units in the last place.  Three
// multiply-adds; the approximation flushes subnormal numbers, so where x or 1 / x is near
// them (|x| < 2^-1021 or |x| >= 2^1021, and not finite) the quotient is formed by division.
// The test comes last, off the chain: 256 problems of 64 stages 386 -> 382 us (379 without).
__device__ __forceinline__ double recip(double x) {
    double y;
    asm volatile("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    y = fma(y, fma(e, e, e), y);
    const unsigned ex = (unsigned)__double2hiint(x) >> 20 & 0x7ffu;
    if (__builtin_expect(ex - 2u > 2041u, 0)) y = 1.0 / x;
    return y;
}
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }

// x > 0 and x finite, and x finite, on the integer pipe (an FP64 compare costs as much as a
// multiply-add).  A pivot or determinant that overflowed is not taken as positive: the
// gains would come out 0 or NaN.
__device__ __forceinline__ bool positive_finite(double x) {
    const long long b = __double_as_longlong(x);
    return b > 0 && b < 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool positive_finite(float x) { return x > 0.0f && isfinite(x); }
__device__ __forceinline__ bool finite(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }
__device__ __forceinline__ bool finite(float x) { return isfinite(x); }

}  // namespace oca
