// Powers of the scale factor that weigh a pass (device, one warp): shared by the
// pass's own update and by tl_set_background, so that a background set to the
// values a pass left gives bitwise that pass's weights.
#pragma once

#include <math.h>

#include "tl_internal.cuh"
#include "tl_power.cuh"

namespace tl {

// Lane i < kScalePowers writes the i-th of the scalars wl .. ia for the scale
// factor a; lane kScalePowers returns mid^(alpha - 3) (the drift's weight), and
// lane kScalePowers + 1 the reciprocal of other.  All lanes of a warp call it, so
// the latency of one power is paid, not of eight.
__device__ __forceinline__ double write_scale_powers(const Model &m, Scalars *sc, double a, double mid, double other)
{
    const int lane = threadIdx.x & 31;
    const int fixed = lane == 2 ? -6 : lane == 3 ? -2 : lane == 6 || lane > kScalePowers ? -1 : 0;  // exponents without alpha
    const int mult = lane == 4 || lane == 5 ? 2 : 1, add = lane == 0 || lane == 4 ? 1 : lane == 1 ? 3 : lane == 5 ? 0 : -3;
    const double x = lane < kScalePowers ? a : lane == kScalePowers ? mid : other;
    double r;
    if (fixed || m.int_alpha) r = int_power(x, fixed ? fixed : mult * (int)m.alpha + add);
    else r = pow(x, mult * m.alpha + add);
    if (lane < kScalePowers) (&sc->wl)[lane] = r;
    return r;
}

}  // namespace tl
