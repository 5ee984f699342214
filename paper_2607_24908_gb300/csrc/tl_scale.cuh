// Powers of the scale factor that weigh a pass (device, one warp): shared by the
// pass's own update and by tl_set_background, so that a background set to the
// values a pass left gives bitwise that pass's weights.
#pragma once

#include <math.h>

#include "tl_internal.cuh"

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

// x^n by repeated squaring of x, or of inv = 1/x for n < 0; |n| <= 16.
__device__ __forceinline__ double int_power(double x, double inv, int n)
{
    double b = n < 0 ? inv : x;
    unsigned k = n < 0 ? -n : n;
    if (k == 0) return 1.0;
    for (; !(k & 1); k >>= 1) b *= b;
    double acc = b;
    while (k >>= 1) {
        b *= b;
        if (k & 1) acc *= b;
    }
    return acc;
}

// Lane i < kScalePowers writes the i-th of the scalars wl .. ia for the scale
// factor a; lane kScalePowers returns mid^(alpha - 3) (the drift's weight), and
// lane kScalePowers + 1 the reciprocal of other.  All lanes of a warp call it, so
// the latency of one power is paid, not of eight.
__device__ __forceinline__ double write_scale_powers(const Model &m, Scalars *sc, double a, double mid, double other)
{
    const int lane = threadIdx.x & 31;
    const int fixed = lane == 2 ? -6 : lane == 3 ? -2 : lane == 6 ? -1 : 0;  // exponents without alpha
    const int mult = lane == 4 || lane == 5 ? 2 : 1, add = lane == 0 || lane == 4 ? 1 : lane == 1 ? 3 : lane == 5 ? 0 : -3;
    const double x = lane < kScalePowers ? a : lane == kScalePowers ? mid : other;
    const double inv = reciprocal(x);
    if (lane > kScalePowers) return inv;
    double r;
    if (fixed) r = int_power(x, inv, fixed);
    else if (m.int_alpha) r = int_power(x, inv, mult * (int)m.alpha + add);
    else r = pow(x, mult * m.alpha + add);
    if (lane < kScalePowers) (&sc->wl)[lane] = r;
    return r;
}

}  // namespace tl
