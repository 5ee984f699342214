// Launchers of the Fourier-space kernels (initial fields, spectra).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "tl_internal.cuh"

namespace tl {

// A real N^3 array is transformed as the complex array c[z][y][x'] = f(2x') + i
// f(2x'+1), x' < N/2: the dense FP64 array itself, read as N x N x N/2 complex
// values, in place.  With C its (unnormalised) transform and k' < N/2 the
// third index, e and o the transforms of the even and odd columns (C = e + i
// o), the field's own modes are
//   F(n) = e(k') + w o(k'),  F(n - N/2) = e(k') - w o(k'),   w = exp(-2 pi i k'/N)
// with e, o = (C(k) +- conj C(-k))/2, (1, 1/i): half the array and about two
// thirds of the time of a real-to-complex transform (256^3: 1.45 against
// 2.27 ms, 192^3 0.65 against 0.93; sizes with large prime factors 5-10%).

// The modes C of a Gaussian random field (see tl_init_spec), for the inverse
// transform.  power: scratch for mode_powers(N) values, or NULL.
constexpr int mode_powers(int N) { return N * N / 4; }
cudaError_t launch_fill_modes(double2 *modes, double *power, int N, double kIR, double A, double m2, int pi_spectrum,
                              int fixed_modulus, uint64_t seed, uint64_t stream, int sm_count, cudaStream_t s);
// The padded array at dst = base + scale * delta (delta dense; may be NULL), ghost rows included.
cudaError_t launch_assemble(int dtype, void *dst, const double *delta, double base, double scale, int N, long long P,
                            long long PP, cudaStream_t s);
// dst = the padded array at src less its offset (tl_offset.cuh), dense, in FP64; *offset = that.
cudaError_t launch_widen(int dtype, double *dst, const void *src, double *offset, int N, long long P, long long PP,
                         cudaStream_t s);
// Shell sums of |F|^2 / N^6, |n| and mode counts from C (accumulated with atomics);
// *mode0 = F(0), which alone is in shell 0.
cudaError_t launch_bin(const double2 *modes, int N, int nbins, double *Psum, double *rsum, unsigned long long *cnt,
                       double *mode0, int sm_count, cudaStream_t s);

}  // namespace tl
