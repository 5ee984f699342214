// Transforms along y and z, the table of roots (see tl_fft.cuh).
#include <math.h>

#include "tl_fft.cuh"
#include "tl_smem.cuh"

namespace tl {

bool fft_supported(int N)
{
    if (N < 64 || N > 1024) return false;
    int m = N;
    while (m % 2 == 0) m /= 2;
    return m == 1 || m == 3 || m == 5;
}

// The N/2 roots exp(-2 pi i m/N) as pairs (c, t).
static void fft_roots(int N, double2 *roots)
{
    const long double step = 2.0L * 3.14159265358979323846264338327950288L / (long double)N;
    for (int i = 0; i < N / 2; ++i) {
        const long double c = cosl(step * i), s = sinl(step * i);
        const bool turned = 8 * i > N && 8 * i < 3 * N;
        // exp(-i x) = cos x (1 - i tan x) = -i sin x (1 + i cot x)
        roots[i].x = (double)(turned ? s : c);
        roots[i].y = (double)(turned ? c / s : -s / c);
    }
}

// The table travels as a kernel's parameter (8 KB at N = 1024, of the 32 KB that one
// may have): copied at the launch, so that the host has nothing to keep or wait for.
constexpr int kMaxRoots = 512;
struct RootTable {
    double2 v[kMaxRoots];
};
__global__ void __launch_bounds__(256) store_roots(double2 *roots, const __grid_constant__ RootTable table, int count)
{
    for (int i = threadIdx.x; i < count; i += 256) roots[i] = table.v[i];
}

cudaError_t launch_fft_roots(int N, double2 *roots, cudaStream_t s)
{
    if (!fft_supported(N) || N / 2 > kMaxRoots) return cudaErrorInvalidValue;
    RootTable t{};
    fft_roots(N, t.v);
    store_roots<<<1, 256, 0, s>>>(roots, t, N / 2);
    return cudaGetLastError();
}

template <int L>
static cudaError_t columns(double2 *data, const double2 *roots, int N, bool z_axis, bool inverse, cudaStream_t s)
{
    using S = FftSplit<L>;
    constexpr size_t smem = S::smem(false);
    if (smem > 48 * 1024) {
        static SmemLimit limit;
        const cudaError_t e = limit.raise(fft_columns<L>, smem);
        if (e != cudaSuccess) return e;
    }
    const unsigned h = (unsigned)N / 2, lines = (unsigned)N * h, inner = z_axis ? lines : h;
    const size_t plane = (size_t)N * h;
    fft_columns<L><<<(lines + S::B - 1) / S::B, S::THREADS, smem, s>>>(data, roots, N / L, lines, inner, plane,
                                                                        z_axis ? plane : h, inverse);
    return cudaGetLastError();
}

cudaError_t launch_fft_columns(double2 *data, const double2 *roots, int N, bool z_axis, bool inverse, cudaStream_t s)
{
    switch (N) {
#define TL_COLUMNS(L) case L: return columns<L>(data, roots, N, z_axis, inverse, s);
        TL_COLUMNS(64) TL_COLUMNS(128) TL_COLUMNS(256) TL_COLUMNS(512) TL_COLUMNS(1024)
        TL_COLUMNS(96) TL_COLUMNS(192) TL_COLUMNS(384) TL_COLUMNS(768)
        TL_COLUMNS(80) TL_COLUMNS(160) TL_COLUMNS(320) TL_COLUMNS(640)
#undef TL_COLUMNS
    }
    return cudaErrorInvalidValue;
}

}  // namespace tl
