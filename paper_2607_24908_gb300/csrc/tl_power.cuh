// Whole powers and reciprocals in FP64 by short chains of dependent operations
// (device; compiled for the host by a test).
#pragma once

namespace tl {

// 1/x by Newton's iteration in its cubic form from an FP32 reciprocal (error
// 2^-23 -> 2^-69): three dependent FP64 operations of 65 clocks each where a
// division took 550.  Outside FP32's comfortable range: the division.
__device__ __forceinline__ double reciprocal(double x)
{
    if (!(x > 1e-30 && x < 1e30)) return 1.0 / x;
    const double y = (double)(1.0f / (float)x), e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// x^n by repeated squaring, |n| <= 16; for n < 0 the reciprocal of the power (the
// power of a rounded reciprocal would carry its error |n| times).
__device__ __forceinline__ double int_power(double x, int n)
{
    unsigned k = n < 0 ? -n : n;
    if (k == 0) return 1.0;
    double b = x;
    for (; !(k & 1); k >>= 1) b *= b;
    double acc = b;
    while (k >>= 1) {
        b *= b;
        if (k & 1) acc *= b;
    }
    return n < 0 ? reciprocal(acc) : acc;
}

}  // namespace tl
