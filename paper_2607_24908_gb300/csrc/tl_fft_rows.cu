// Transforms along x, between a field and its modes (see tl_fft.cuh).
#include "tl_fft.cuh"
#include "tl_smem.cuh"

namespace tl {

template <int L>
static cudaError_t rows(double2 *data, const FieldRows &field, const double2 *roots, bool inverse, cudaStream_t s)
{
    using S = FftSplit<L>;
    constexpr size_t smem = S::smem(true);
    if (smem > 48 * 1024) {
        static SmemLimit limit;
        const cudaError_t e = limit.raise(fft_rows<L>, smem);
        if (e != cudaSuccess) return e;
    }
    const unsigned lines = (unsigned)field.N * (unsigned)field.N;
    fft_rows<L><<<(lines + S::B - 1) / S::B, S::THREADS, smem, s>>>(data, field, roots, field.N / L, lines, inverse);
    return cudaGetLastError();
}

cudaError_t launch_fft_rows(double2 *data, const FieldRows &field, const double2 *roots, bool inverse, cudaStream_t s)
{
    switch (field.N / 2) {
#define TL_ROWS(L) case L: return rows<L>(data, field, roots, inverse, s);
        TL_ROWS(32) TL_ROWS(64) TL_ROWS(128) TL_ROWS(256) TL_ROWS(512)
        TL_ROWS(48) TL_ROWS(96) TL_ROWS(192) TL_ROWS(384)
        TL_ROWS(40) TL_ROWS(80) TL_ROWS(160) TL_ROWS(320)
#undef TL_ROWS
    }
    return cudaErrorInvalidValue;
}

}  // namespace tl
