// FP64 complex transforms of N x N x N/2 values in place (tl_fourier.cuh says
// what they hold), axis by axis, for N = 2^m, 3 2^m and 5 2^m from 64 to 1024.
//
// What bounds them is the FP64 pipe: a warp's FP64 instruction holds it for 16
// clocks, in which the SM issues up to 64 others, and an axis of 256 points needs
// about seven times as long there as for its memory traffic.  So all that counts
// is the number of FP64 instructions:
//  * a butterfly a +- w b with w = c (1 + i t) (or -i c (1 + i t), whichever has
//    |t| <= 1) takes six fused multiply-adds, two for (1 + i t) b and four for
//    a +- c (...), instead of eight (E. Linzer, E. Feig, "Implementation of efficient
//    FFT algorithms on fused multiply-add architectures", IEEE Trans. Signal
//    Processing 41, 1993); the plain ones (w = 1, -i) take four;
//  * roots come from a table, index work, selects, signs and the exchange through
//    shared memory are other pipes' work and next to free;
//  * FP32 fields are widened by integer instructions (tl_bits.cuh) as they are
//    loaded, and scaled, narrowed and stored by the last pass, which saves a pass
//    over memory on either side.
// 256^3: 340 instructions for 16 points of y or z, 292 for 16 of x and 32 for the
// field's offset (tl_offset.cuh) or, inverse, its scale; the pipe is busy 94% of the
// time.  Against cuFFT (us): y or z 439 -> 305, x 501 + 36 for a pass that widened ->
// 270 (300 with the offset, with which the spectra below take 3% more), inverse x 501 + 70 for one that stored
// -> 298.  A spectrum / an initial field (us, cuFFT -> here): 64^3 106 / 95 -> 100 /
// 89, 96^3 149 / 177 -> 121 / 155, 128^3 277 / 351 -> 206 / 280, 160^3 510 / 643 ->
// 375 / 507, 192^3 774 / 1039 -> 537 / 765, 256^3 1674 / 2204 -> 1134 / 1625, 512^3
// 16881 / 20520 -> 9570 / 13160, 640^3 38440 / 45639 -> 23107 / 30274.  Below 64^3 a
// line has too few threads and cuFFT is faster (48^3 88 / 76 against 112 /
// 97); above 1024 the lines of a CTA do not fit its shared memory.
//
// A line of L points belongs to L/E threads of E points each.  Phase by phase
// (radices R with product L) each thread transforms E/R sets of R points, input
// n = s + i L/R, whose twiddles w_{PR}^{ik}, k = s mod P (P the product of the
// radices before), are part of the radix-2 levels of the set's transform, and
// writes point i to (s - k) R + k + i P: the order comes out right after the last.
// Any factor of 3 or 5 is taken by the first phase, which has no twiddles.
#pragma once

#include <cuda_runtime.h>

#include "tl_bits.cuh"
#include "tl_internal.cuh"
#include "tl_offset.cuh"

namespace tl {

// Radices and threads of a line of L points.
template <int L>
struct FftSplit {
    static constexpr int ODD = L % 3 == 0 ? 3 : L % 5 == 0 ? 5 : 1;
    static constexpr int E = ODD == 1 ? 16 : ODD == 3 ? 24 : 20;  // points per thread
    static constexpr int T = L / E;                               // threads per line
    static constexpr int R2 = ODD == 1 ? (T <= 16 ? T : T == 32 ? 8 : 16) : ODD == 3 ? (T <= 8 ? T : 8) : (T <= 4 ? T : 4);
    static constexpr int R3 = T / R2 <= 4 ? T / R2 : 4;
    static constexpr int R4 = T / R2 / R3;
    static_assert(E * R2 * R3 * R4 == L && T > 1, "radices");
    // lines per CTA: 128 threads at least, rows of 8 neighbouring columns (128 bytes)
    static constexpr int B = T * 8 >= 128 ? (T * 8 > 256 ? (T * 4 > 256 ? 2 : 4) : 8) : 128 / T;
    static constexpr int THREADS = T * B;
    static constexpr int PITCH = L + L / 16 + 1;  // of a line in shared memory (rows)
    static constexpr size_t smem(bool rows) { return (size_t)B * (rows ? PITCH : L) * sizeof(double2); }
    static constexpr int MINB = ODD == 3 ? 384 / THREADS : 512 / THREADS;  // 168 or 128 registers
};

// Where a factor's index lies in [0, L/2) of the half circle: whether |sin| > |cos|.
template <int L>
__device__ __forceinline__ bool root_turned(int idx)
{
    return 8 * idx > L && 8 * idx < 3 * L;
}

// (a, o) <- (a + w o, a - w o), w = exp(-2 pi i idx/L) (times -i: quarter), root = its
// (c, t): w = c (1 + i t), or, turned, w = -i c (1 + i t).
__device__ __forceinline__ void fma_butterfly(double2 &a, double2 &o, double2 root, bool turned, bool quarter)
{
    // -i (x + i y) = y - i x: swapped parts u, v = y, x stand for u - i v
    const bool s = turned != quarter;
    const double u = s ? o.y : o.x, v = s ? o.x : o.y;
    const double t = flip(root.y, s);
    const double x = __fma_rn(-t, v, u), y = __fma_rn(t, u, v);
    // turned twice: -1
    const double cx = flip(root.x, turned && quarter), cy = flip(cx, s);
    const double ax = a.x, ay = a.y;
    a.x = __fma_rn(cx, x, ax);
    a.y = __fma_rn(cy, y, ay);
    o.x = __fma_rn(-cx, x, ax);
    o.y = __fma_rn(-cy, y, ay);
}

__device__ __forceinline__ void plain_butterfly(double2 &a, double2 &o)
{
    const double2 b = o;
    o = make_double2(a.x - b.x, a.y - b.y);
    a = make_double2(a.x + b.x, a.y + b.y);
}

__device__ __forceinline__ void quarter_butterfly(double2 &a, double2 &o)  // w = -i
{
    const double2 b = o;
    o = make_double2(a.x - b.y, a.y + b.x);
    a = make_double2(a.x + b.y, a.y - b.x);
}

__device__ __forceinline__ void dft3(double2 &a, double2 &b, double2 &c)
{
    const double h = 0.86602540378443864676;  // sin(2 pi/3)
    const double sx = b.x + c.x, sy = b.y + c.y, dx = b.x - c.x, dy = b.y - c.y;
    const double mx = __fma_rn(-0.5, sx, a.x), my = __fma_rn(-0.5, sy, a.y);
    a = make_double2(a.x + sx, a.y + sy);
    b = make_double2(__fma_rn(h, dy, mx), __fma_rn(-h, dx, my));
    c = make_double2(__fma_rn(-h, dy, mx), __fma_rn(h, dx, my));
}

__device__ __forceinline__ void dft5(double2 &a, double2 &b, double2 &c, double2 &d, double2 &e)
{
    const double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;  // cos(2 pi/5), cos(4 pi/5)
    const double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;   // sin(2 pi/5), sin(4 pi/5)
    const double px = b.x + e.x, py = b.y + e.y, qx = c.x + d.x, qy = c.y + d.y;
    const double ux = b.x - e.x, uy = b.y - e.y, vx = c.x - d.x, vy = c.y - d.y;
    const double m1x = __fma_rn(c1, px, __fma_rn(c2, qx, a.x)), m1y = __fma_rn(c1, py, __fma_rn(c2, qy, a.y));
    const double m2x = __fma_rn(c2, px, __fma_rn(c1, qx, a.x)), m2y = __fma_rn(c2, py, __fma_rn(c1, qy, a.y));
    const double n1x = __fma_rn(s1, ux, s2 * vx), n1y = __fma_rn(s1, uy, s2 * vy);
    const double n2x = __fma_rn(s2, ux, -(s1 * vx)), n2y = __fma_rn(s2, uy, -(s1 * vy));
    a = make_double2(a.x + px + qx, a.y + py + qy);
    b = make_double2(m1x + n1y, m1y - n1x);  // m1 - i n1
    e = make_double2(m1x - n1y, m1y + n1x);
    c = make_double2(m2x + n2y, m2y - n2x);
    d = make_double2(m2x - n2y, m2y + n2x);
}

// Where input i of a set of R points is held: the levels of radix 2 take their
// input in bit-reversed order, each ODD points of the base in a row.
template <int R, int ODD>
__host__ __device__ constexpr int fft_slot(int i)
{
    constexpr int M = R / ODD;
    int b = 0;
    for (int bit = 1, j = i % M; bit < M; bit *= 2, j /= 2) b = 2 * b + j % 2;
    return b * ODD + i / M;
}

// Transform of R points in registers, in place, twiddled by k (0 <= k < P).
template <int L, int R, int ODD, int P>
__device__ __forceinline__ void fft_set(double2 *v, int k, const double2 *__restrict__ roots, int mul)
{
    constexpr int M = R / ODD;
#pragma unroll
    for (int b = 0; b < M; ++b) {
        if (ODD == 3) dft3(v[3 * b], v[3 * b + 1], v[3 * b + 2]);
        if (ODD == 5) dft5(v[5 * b], v[5 * b + 1], v[5 * b + 2], v[5 * b + 3], v[5 * b + 4]);
    }
#pragma unroll
    for (int lev = 1; lev <= 4; ++lev) {
        const int h = ODD << lev;
        if (h > R) continue;
        const bool halves = h % 4 == 0;  // w^(q + h/4) = -i w^q
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            if (q >= (halves ? h / 4 : h / 2)) continue;
            const bool one = P == 1 && q == 0;
            const int idx = (k + P * q) * (L / (P * h));
            double2 root = make_double2(1.0, 0.0);
            if (!one) root = __ldg(roots + idx * mul);
            const bool turned = root_turned<L>(idx);
#pragma unroll
            for (int b = 0; b < R; ++b) {
                if (b % h) continue;
                if (one) plain_butterfly(v[b + q], v[b + q + h / 2]);
                else fma_butterfly(v[b + q], v[b + q + h / 2], root, turned, false);
                if (halves) {
                    const int q2 = q + h / 4;
                    if (one) quarter_butterfly(v[b + q2], v[b + q2 + h / 2]);
                    else fma_butterfly(v[b + q2], v[b + q2 + h / 2], root, turned, true);
                }
            }
        }
    }
}

// One phase: E/R sets of the thread, input by load(n), output by store(n, value).
// sync: between the loads and the stores (both in shared memory).
template <int L, int R, int ODD, int P, bool SYNC, typename Load, typename Store>
__device__ __forceinline__ void fft_phase(int j, const double2 *__restrict__ roots, int mul, Load load, Store store)
{
    using S = FftSplit<L>;
    constexpr int SETS = S::E / R;
    double2 v[S::E];
#pragma unroll
    for (int u = 0; u < SETS; ++u)
#pragma unroll
        for (int i = 0; i < R; ++i) v[u * R + fft_slot<R, ODD>(i)] = load(j + u * S::T + i * (L / R));
#pragma unroll
    for (int u = 0; u < SETS; ++u) fft_set<L, R, ODD, P>(v + u * R, (j + u * S::T) % P, roots, mul);
    if (SYNC) __syncthreads();
#pragma unroll
    for (int u = 0; u < SETS; ++u) {
        const int s = j + u * S::T, k = s % P;
#pragma unroll
        for (int i = 0; i < R; ++i) store((s - k) * R + k + i * P, v[u * R + i]);
    }
    if (SYNC) __syncthreads();
}

// All phases of a line: input by load, output by store, between them ex(n), the
// line's places in shared memory.
template <int L, typename Load, typename Store, typename Ex>
__device__ __forceinline__ void fft_line(int j, const double2 *__restrict__ roots, int mul, Load load, Store store, Ex ex)
{
    using S = FftSplit<L>;
    auto put = [&](int n, double2 v) { *ex(n) = v; };
    auto get = [&](int n) { return *ex(n); };
    fft_phase<L, S::E, S::ODD, 1, true>(j, roots, mul, load, put);
    if constexpr (S::R3 == 1) {
        fft_phase<L, S::R2, 1, S::E, false>(j, roots, mul, get, store);
    } else {
        fft_phase<L, S::R2, 1, S::E, true>(j, roots, mul, get, put);
        if constexpr (S::R4 == 1) {
            fft_phase<L, S::R3, 1, S::E * S::R2, false>(j, roots, mul, get, store);
        } else {
            fft_phase<L, S::R3, 1, S::E * S::R2, true>(j, roots, mul, get, put);
            fft_phase<L, S::R4, 1, S::E * S::R2 * S::R3, false>(j, roots, mul, get, store);
        }
    }
}

// The inverse transform is the forward one of values with exchanged parts.
__device__ __forceinline__ double2 parts(double2 v, bool exchange) { return exchange ? make_double2(v.y, v.x) : v; }

// Lines along y or z, in place: line l has its points `stride` apart from
// (l / inner) outer + l mod inner.  roots: exp(-2 pi i m/N) as (c, t), mul = N/L.
template <int L>
__global__ void __launch_bounds__(FftSplit<L>::THREADS, FftSplit<L>::MINB)
    fft_columns(double2 *data, const double2 *__restrict__ roots, int mul, unsigned lines, unsigned inner, size_t outer,
                size_t stride, bool inverse)
{
    using S = FftSplit<L>;
    extern __shared__ double2 sh[];
    const int lane = threadIdx.x % S::B, j = threadIdx.x / S::B;
    const unsigned l = blockIdx.x * S::B + lane;
    const bool active = l < lines;
    double2 *p = data + (l / inner) * outer + l % inner;
    fft_line<L>(
        j, roots, mul, [&](int n) { return active ? parts(p[n * stride], inverse) : make_double2(0.0, 0.0); },
        [&](int n, double2 v) {
            if (active) p[n * stride] = parts(v, inverse);
        },
        [&](int n) { return sh + n * S::B + lane; });
}

struct FieldRows {  // a padded field array, rows of N sites
    void *p;
    int f32;
    int N;
    long long pitch, pplane;
    double base, scale;    // inverse: site = base + scale value
    double *offset;        // forward: value = site - offset, which is left here (tl_offset.cuh)
};

// Lines along x, of L = N/2 points: forward from a field (sites 2n and 2n + 1 the
// parts of point n) to modes, inverse from modes to a field with its ghost rows.
template <int L>
__global__ void __launch_bounds__(FftSplit<L>::THREADS, FftSplit<L>::MINB)
    fft_rows(double2 *data, FieldRows field, const double2 *__restrict__ roots, int mul, unsigned lines, bool inverse)
{
    using S = FftSplit<L>;
    extern __shared__ double2 sh[];
    const int row = threadIdx.x / S::T, j = threadIdx.x % S::T;
    const unsigned l = blockIdx.x * S::B + row;
    const bool active = l < lines;
    const int z = l / (unsigned)field.N, y = l % (unsigned)field.N;
    const long long at = z * field.pplane + y * field.pitch;
    double2 *p = data + (size_t)l * L;
    double off = 0.0;
    if (!inverse) {
        off = field.f32 ? field_offset(static_cast<const float *>(field.p), field.N, field.pitch, field.pplane)
                        : field_offset(static_cast<const double *>(field.p), field.N, field.pitch, field.pplane);
        if (blockIdx.x == 0 && threadIdx.x == 0) *field.offset = off;
    }
    fft_line<L>(
        j, roots, mul,
        [&](int n) {
            if (!active) return make_double2(0.0, 0.0);
            if (inverse) return parts(p[n], true);
            if (!field.f32) {
                const double2 v = *reinterpret_cast<const double2 *>(static_cast<const double *>(field.p) + at + 2 * n);
                return make_double2(v.x - off, v.y - off);
            }
            const float2 v = *reinterpret_cast<const float2 *>(static_cast<const float *>(field.p) + at + 2 * n);
            return make_double2(widen_bits(v.x) - off, widen_bits(v.y) - off);
        },
        [&](int n, double2 v) {
            if (!active) return;
            if (!inverse) {
                p[n] = v;
                return;
            }
            const double a = field.base + field.scale * v.y, b = field.base + field.scale * v.x;
            const long long ghost = y == 0 ? field.N * field.pitch : y == field.N - 1 ? -(field.N * field.pitch) : 0;
            if (field.f32) {
                float *o = static_cast<float *>(field.p) + at + 2 * n;
                *reinterpret_cast<float2 *>(o) = make_float2(narrow_bits(a), narrow_bits(b));
                if (ghost) *reinterpret_cast<float2 *>(o + ghost) = make_float2(narrow_bits(a), narrow_bits(b));
            } else {
                double *o = static_cast<double *>(field.p) + at + 2 * n;
                *reinterpret_cast<double2 *>(o) = make_double2(a, b);
                if (ghost) *reinterpret_cast<double2 *>(o + ghost) = make_double2(a, b);
            }
        },
        [&](int n) { return sh + row * S::PITCH + n + n / 16; });
}

// N that the kernels above take (else a library transform).
bool fft_supported(int N);
// Write the table of N/2 roots exp(-2 pi i m/N), as pairs (c, t), to the device; only enqueues.
cudaError_t launch_fft_roots(int N, double2 *roots, cudaStream_t s);
cudaError_t launch_fft_columns(double2 *data, const double2 *roots, int N, bool z_axis, bool inverse, cudaStream_t s);
cudaError_t launch_fft_rows(double2 *data, const FieldRows &field, const double2 *roots, bool inverse, cudaStream_t s);

}  // namespace tl
