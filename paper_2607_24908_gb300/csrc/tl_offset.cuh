// The constant that is taken off a field before its spectrum's transform.
//
// The even and odd columns are summed apart (tl_fourier.cuh), so that with a mean m
// every row's sums carry roundings of N m/2, which the difference that gives the modes
// nx = N/2 does not cancel: the corner mode (N/2, N/2, N/2) of a field of mean 5 sigma
// was off by 3e-14 (128^3) and 1.1e-13 (160^3) of its power, a real-to-complex
// transform's by 4e-15 and 7e-15.  Less a constant near the mean, which mode 0 gets
// back, it is off by 5e-15 and 4e-15, and all shells by 5e-16 and 4e-16 (rms), where
// that transform was off by 1.0e-15 and 1.3e-15.
//
// The constant is the median of nine sites spread over the lattice: a field without a
// mean loses nothing to it, and lumps do not move it.  Every warp forms it for itself
// with integer instructions (the transform's kernels wait for the FP64 pipe; a kernel
// of its own took 3 to 9 us), and a site costs one FP64 addition: a spectrum of 256^3
// 1112 -> 1144 us, of 128^3 195 both.
#pragma once

#include "tl_bits.cuh"

namespace tl {

__device__ __forceinline__ double as_double(float v) { return widen_bits(v); }
__device__ __forceinline__ double as_double(double v) { return v; }

// In every lane of a whole warp; 0 if the median is not finite.
template <typename T>
__device__ __forceinline__ double field_offset(const T *src, int N, long long P, long long PP)
{
    const int i = threadIdx.x & 31;
    double v = 0.0;
    if (i < 9) v = as_double(src[(long long)(i * N / 9) * PP + (long long)(4 * i % 9 * N / 9) * P + 7 * i % 9 * N / 9]);
    const long long bits = __double_as_longlong(v), key = bits ^ (bits < 0 ? 0x7fffffffffffffffll : 0);  // in order of v
    int below = 0;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const long long u = __shfl_sync(0xffffffffu, key, j);
        below += u < key || (u == key && j < i);
    }
    const bool finite = (bits & 0x7ff0000000000000ll) != 0x7ff0000000000000ll;
    const unsigned median = __ballot_sync(0xffffffffu, i < 9 && below == 4 && finite);
    return median ? __shfl_sync(0xffffffffu, v, __ffs(median) - 1) : 0.0;
}

}  // namespace tl
