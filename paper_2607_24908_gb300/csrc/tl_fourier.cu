// Initial Gaussian random fields and binned power spectra (off the per-step
// loop).  The paper prepares states and measures in Fourier space through its
// automatic Fourier views (Sec. 2) with Philox-2x64 random numbers (Sec. 2);
// here the mode draw, the field assembly and the shell binning are kernels
// of this library; the transforms (FP64, complex, of half the real size:
// tl_fourier.cuh) are its own for the sizes of tl_fft.cuh, cuFFT library calls
// for the others.
#include <math.h>

#include "tl_bits.cuh"
#include "tl_boxmuller.cuh"
#include "tl_fourier.cuh"
#include "tl_offset.cuh"
#include "tl_philox.cuh"
#include "tl_smem.cuh"

namespace tl {

__device__ __forceinline__ int signed_mode(int i, int N) { return (i < N / 2) ? i : i - N; }

// exp(sign 2 pi i j/N), j = 0 .. N/4, into a CTA's shared table.
__device__ __forceinline__ void fill_roots(double2 *root, int N, double sign)
{
    for (int j = threadIdx.x; j <= N / 4; j += blockDim.x) {
        double s, c;
        sincospi(2.0 * (double)j / (double)N, &s, &c);
        root[j] = make_double2(c, sign * s);
    }
    __syncthreads();
}

struct ModeSpec {
    int N;
    double kIR2, m2, amp2;  // amp2 = A/(2 L^3)
    int pi_spectrum, fixed_modulus;
    uint64_t seed, stream;
};

// The mode n = (nx, iy, iz) (nx >= 0 itself, iy and iz array indices): modulus
// sqrt(P/L^3) times the Rayleigh factor sqrt(-ln u1), phase 2 pi u2, drawn at
// the member of each Hermitian pair with the first nonzero of (nx, ny, nz)
// positive; zero outside 0 < |n| < N/2.
__device__ __forceinline__ double mode_power(const ModeSpec &p, int r2)  // P/L^3, r2 = |n|^2
{
    const double om2 = p.kIR2 * (double)r2 + p.m2;
    return p.amp2 * (p.pi_spectrum ? sqrt(om2) : rsqrt(om2));
}

__global__ void __launch_bounds__(256) mode_power_kernel(double *power, int count, ModeSpec p)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < count) power[i] = i ? mode_power(p, i) : 0.0;
}

__device__ __forceinline__ double2 draw_mode(const BoxMullerTable *t, const double *__restrict__ power, const ModeSpec &p,
                                             int nx, int iy, int iz)
{
    const int N = p.N;
    const int ny = signed_mode(iy, N), nz = signed_mode(iz, N);
    const int r2 = nx * nx + ny * ny + nz * nz;  // N <= 2048: below 2^22
    if (r2 == 0 || 4 * r2 >= N * N) return make_double2(0.0, 0.0);
    const bool canon = nx > 0 || ny > 0 || (ny == 0 && nz > 0);
    const int dy = canon ? iy : (iy ? N - iy : 0), dz = canon ? iz : (iz ? N - iz : 0);
    uint64_t w0, w1;
    philox2x64_10(((uint64_t)dz * N + (uint64_t)dy) * N + (uint64_t)nx, p.stream, p.seed, w0, w1);
    const double P = power ? __ldg(power + r2) : mode_power(p, r2);
    const double amp = sqrt(p.fixed_modulus ? P : P * neg_log_u53(t, (w0 >> 11) + 1));
    double s, c;
    unit_circle_u53(t, w1 >> 11, c, s);
    return make_double2(amp * c, canon ? amp * s : -amp * s);
}

// One thread per row (iz, iy) and k = 0 .. N/4: the modes F1 = F(k, row) and
// F2 = F(N/2 - k, -row) together give C(k, row) = S + Z and C(N/2 - k, -row) =
// conj(S - Z) with S = F1 + conj F2, Z = i exp(2 pi i k/N) (F1 - conj F2).  At
// k = 0 the partner mode (nx = N/2) is zero and so is the second value's
// entry; at k = N/4 both threads of a pair of rows write their own.
//
// Bound by the FP64 pipe: one square root of the whole modulus squared instead
// of four roots and two divisions, 256^3 1305 -> 996 us a field, and the table
// form of the logarithm and the circle (tl_boxmuller.cuh), 996 -> 610 us; P by |n|^2
// from a table that a small kernel fills first (a root and three operations a mode
// less, the same values) and integer-to-FP64 conversions by bits, 604 -> 512 us; four
// operations a draw for its last roundings, 512 -> 555.
__global__ void __launch_bounds__(256) fill_modes_kernel(double2 *modes, const double *__restrict__ power, ModeSpec p)
{
    extern __shared__ double2 root[];
    __shared__ BoxMullerTable table;
    const int N = p.N, h = N / 2, q = N / 4 + 1;
    load_box_muller(&table);
    fill_roots(root, N, 1.0);
    const unsigned total = (unsigned)N * N * q;  // N <= 2048: below 2^32
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < total; i += gridDim.x * 256u) {
        const unsigned row = i / q, k = i - row * q;
        const int iz = row / N, iy = row - (unsigned)iz * N;
        const int my = iy ? N - iy : 0, mz = iz ? N - iz : 0;
        const double2 a = draw_mode(&table, power, p, k, iy, iz);
        if (k == 0) {  // (1 + i) F1
            modes[(size_t)row * h] = make_double2(a.x - a.y, a.x + a.y);
            continue;
        }
        const double2 b = draw_mode(&table, power, p, h - k, my, mz);
        const double2 w = root[k];
        const double dx = a.x - b.x, dy = a.y + b.y;
        const double zx = -(w.x * dy + w.y * dx), zy = w.x * dx - w.y * dy;
        const double sx = a.x + b.x, sy = a.y - b.y;
        modes[(size_t)row * h + k] = make_double2(sx + zx, sy + zy);
        if (4 * (int)k != N) modes[((size_t)mz * N + my) * h + (h - k)] = make_double2(sx - zx, zy - sy);
    }
}

// Four consecutive sites per thread (a row starts a 128-byte line in both
// layouts' FP32 form and N is a multiple of 4): 16- and 32-byte accesses, one
// index decomposition for the four.  Conversions are integer instructions
// (tl_bits.cuh; a field without fluctuations is converted once, on the host): us,
// 256^3 FP32, with F2F -> without: fill 69 -> 18.
template <typename T>
struct Four;
template <>
struct Four<float> {
    static __device__ __forceinline__ void ld(const float *p, double (&v)[4])
    {
        const float4 a = *reinterpret_cast<const float4 *>(p);
        v[0] = widen_bits(a.x), v[1] = widen_bits(a.y), v[2] = widen_bits(a.z), v[3] = widen_bits(a.w);
    }
    static __device__ __forceinline__ void fill(float *p, float v) { *reinterpret_cast<float4 *>(p) = make_float4(v, v, v, v); }
    static __device__ __forceinline__ void st(float *p, const double (&v)[4])
    {
        *reinterpret_cast<float4 *>(p) = make_float4(narrow_bits(v[0]), narrow_bits(v[1]), narrow_bits(v[2]), narrow_bits(v[3]));
    }
};
template <>
struct Four<double> {
    static __device__ __forceinline__ void ld(const double *p, double (&v)[4])
    {
        const double2 a = *reinterpret_cast<const double2 *>(p), b = *reinterpret_cast<const double2 *>(p + 2);
        v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
    }
    static __device__ __forceinline__ void fill(double *p, double v)
    {
        *reinterpret_cast<double2 *>(p) = make_double2(v, v);
        *reinterpret_cast<double2 *>(p + 2) = make_double2(v, v);
    }
    static __device__ __forceinline__ void st(double *p, const double (&v)[4])
    {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2 *>(p + 2) = make_double2(v[2], v[3]);
    }
};

template <typename T>
__global__ void __launch_bounds__(256) assemble_kernel(T *dst, const double *delta, double base, T base_t, double scale,
                                                       int N, long long P, long long PP)
{
    const unsigned quads = (unsigned)N / 4, i = blockIdx.x * 256u + threadIdx.x;
    const unsigned row = i / quads, x = 4 * (i - row * quads);
    const int z = row / N, y = row - (unsigned)z * N;
    if (z >= N) return;
    T *out = dst + z * PP + y * P + x;
    const long long ghost = y == 0 ? (long long)N * P : y == N - 1 ? -((long long)N * P) : 0;  // to the ghost row
    if (!delta) {
        Four<T>::fill(out, base_t);
        if (ghost) Four<T>::fill(out + ghost, base_t);
        return;
    }
    double v[4];
    Four<double>::ld(delta + (size_t)row * N + x, v);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = base + scale * v[j];
    Four<T>::st(out, v);
    if (ghost) Four<T>::st(out + ghost, v);
}

template <typename T>
__global__ void __launch_bounds__(256)
    widen_kernel(double *dst, const T *src, double *offset, int N, long long P, long long PP)
{
    const double off = field_offset(src, N, P, PP);
    if (blockIdx.x == 0 && threadIdx.x == 0) *offset = off;
    const unsigned quads = (unsigned)N / 4, i = blockIdx.x * 256u + threadIdx.x;
    const unsigned row = i / quads, x = 4 * (i - row * quads);
    const int z = row / N, y = row - (unsigned)z * N;
    if (z >= N) return;
    double v[4];
    Four<T>::ld(src + z * PP + y * P + x, v);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] -= off;
    Four<double>::st(dst + (size_t)row * N + x, v);
}

// bin(s) = floor(sqrt(s) + 1/2) for an integer 0 <= s < 2^24 and root = sqrt(s)
// to FP32, decided in integers: m is the bin iff m (m - 1) < s <= m (m + 1).
__device__ __forceinline__ int shell_bin(int s, float root)
{
    int m = (int)(root + 0.5f);
    while (m > 0 && m * (m - 1) >= s) --m;
    while ((m + 1) * m < s) ++m;
    return m;
}

// sqrt(s) in FP64 from its FP32 value r: two terms of the Taylor series of the
// root about r^2 (r is right to 2^-24, so the next term is below 2^-70).
__device__ __forceinline__ double refine_root(int s, float root)
{
    if (s == 0) return 0.0;
    const double r = (double)root, h = (double)(0.5f / root);
    const double d = fma(-r, r, (double)s);
    const double e = d * fma(-fma(2.0 * r, h, -1.0), h, h);  // d/(2r), h refined once
    return fma(-e * e, h, r + e);
}

// Adds (P, r, w) to the shell sums of bin b: runs of lanes with the same bin
// are summed first (a segmented sum towards each run's first lane), so that a
// warp's atomics mostly go to different bins.
__device__ __forceinline__ void add_to_shell(int b, double P, double r, unsigned w, double *sP, double *sR,
                                             unsigned long long *sC)
{
    const int lane = threadIdx.x & 31;
    const bool head = __shfl_up_sync(0xffffffffu, b, 1) != b || lane == 0;
    const unsigned above = (0xfffffffeu << lane) & __ballot_sync(0xffffffffu, head);
    const int end = above ? __ffs(above) - 1 : 32;  // the run's end
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double oP = __shfl_down_sync(0xffffffffu, P, o), oR = __shfl_down_sync(0xffffffffu, r, o);
        const unsigned ow = __shfl_down_sync(0xffffffffu, w, o);
        if (lane + o < end) P += oP, r += oR, w += ow;
    }
    if (w && head) {
        atomicAdd(sP + b, P);
        atomicAdd(sR + b, r);
        atomicAdd(sC + b, (unsigned long long)w);
    }
}

// One thread per (a, b, k), N/2 >= a >= b >= 0, k = 0 .. N/4: the modes |nx| = k
// and |nx| = N/2 - k of the up to eight rows (+-a, +-b), (+-b, +-a), which
// share their shells, are summed in registers before they reach the shell
// sums.  Each C is read once, 16 reads of a thread in flight.
//
// FP64-pipe work a mode: 8 operations for |F|^2 and its sum.  With one shared
// FP64 atomic (a compare-and-swap loop) for each of a mode's three sums this
// took 475 us at 256^3; here 193.
__global__ void __launch_bounds__(256) bin_kernel(const double2 *__restrict__ modes, int N, int nbins, double *Psum,
                                                  double *rsum, unsigned long long *cnt, double *mode0)
{
    extern __shared__ double2 root[];  // N/4 + 1 roots, then the CTA's shell sums
    const int h = N / 2, q = N / 4 + 1;
    double *sP = reinterpret_cast<double *>(root + q);
    double *sR = sP + nbins;
    unsigned long long *sC = reinterpret_cast<unsigned long long *>(sR + nbins);
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
        sP[b] = 0.0;
        sR[b] = 0.0;
        sC[b] = 0ull;
    }
    fill_roots(root, N, -1.0);  // and a barrier
    if (blockIdx.x == 0 && threadIdx.x == 0) *mode0 = modes[0].x + modes[0].y;
    const unsigned pairs = (unsigned)(h + 1) * (h + 2) / 2, total = pairs * (unsigned)q;  // below 2^29
    const double scale = 0.25 / ((double)N * N * N) / ((double)N * N * N);
    for (unsigned first = blockIdx.x * 256u; first < total; first += gridDim.x * 256u) {
        const unsigned i = first + threadIdx.x;
        const bool active = i < total;
        const unsigned pair = active ? i / q : 0;
        const int k = active ? (int)(i - pair * q) : 0;
        int a = (int)((sqrtf(8.0f * (float)pair + 1.0f) - 1.0f) * 0.5f);  // pair = a (a + 1)/2 + b
        while ((unsigned)(a + 1) * (a + 2) / 2 <= pair) ++a;
        while ((unsigned)a * (a + 1) / 2 > pair) --a;
        const int b = (int)(pair - (unsigned)a * (a + 1) / 2);
        const double2 w = root[k];
        const int kp = k ? h - k : 0;
        double P1 = 0.0, P2 = 0.0;
        unsigned rows = 0;
        if (active) {
            double2 c[8], d[8];
            bool own[8];
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const int vy = v & 1 ? b : a, vz = v & 1 ? a : b;
                const bool ny = v & 2, nz = v & 4;  // the negative one
                own[v] = !(((v & 1) && a == b) || (ny && (vy == 0 || vy == h)) || (nz && (vz == 0 || vz == h)));
                const int iy = ny && vy ? N - vy : vy, iz = nz && vz ? N - vz : vz;
                const int my = iy ? N - iy : 0, mz = iz ? N - iz : 0;
                c[v] = __ldg(modes + ((size_t)iz * N + iy) * h + k);
                d[v] = __ldg(modes + ((size_t)mz * N + my) * h + kp);
            }
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                if (!own[v]) continue;  // a row already among the others
                const double ex = c[v].x + d[v].x, ey = c[v].y - d[v].y, fx = c[v].x - d[v].x, fy = c[v].y + d[v].y;
                const double gx = fma(w.x, fy, w.y * fx), gy = fma(w.y, fy, -(w.x * fx));  // -i w (fx + i fy)
                const double px = ex + gx, py = ey + gy, mx = ex - gx, mmy = ey - gy;
                P1 = fma(px, px, fma(py, py, P1));
                P2 = fma(mx, mx, fma(mmy, mmy, P2));
                ++rows;
            }
        }
        // |nx| = k, both signs of it (0 once); |nx| = N/2 - k, both signs (N/2
        // once, N/4 counted as k)
        const unsigned m1 = k ? 2u : 1u, m2 = k == 0 ? 1u : 4 * k == N ? 0u : 2u;
        const int s = a * a + b * b, s1 = s + k * k, s2 = s + (h - k) * (h - k);
        const float r1 = sqrtf((float)s1), r2 = sqrtf((float)s2);
        add_to_shell(shell_bin(s1, r1), (double)m1 * scale * P1, (double)(m1 * rows) * refine_root(s1, r1), m1 * rows,
                     sP, sR, sC);
        add_to_shell(shell_bin(s2, r2), (double)m2 * scale * P2, (double)(m2 * rows) * refine_root(s2, r2), m2 * rows,
                     sP, sR, sC);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
        if (sC[b]) {
            atomicAdd(&Psum[b], sP[b]);
            atomicAdd(&rsum[b], sR[b]);
            atomicAdd(&cnt[b], sC[b]);
        }
    }
}

static unsigned grid_for(size_t n, int sm_count, int per_sm)
{
    const size_t g = (n + 255) / 256, cap = (size_t)(sm_count > 0 ? sm_count : 152) * per_sm;
    return (unsigned)(g < cap ? g : cap);
}

cudaError_t launch_fill_modes(double2 *modes, double *power, int N, double kIR, double A, double m2, int pi_spectrum,
                              int fixed_modulus, uint64_t seed, uint64_t stream, int sm_count, cudaStream_t s)
{
    const double L = 2.0 * M_PI / kIR;
    const ModeSpec p{N, kIR * kIR, m2, A / (2.0 * L * L * L), pi_spectrum, fixed_modulus, seed, stream};
    const size_t total = (size_t)N * N * (N / 4 + 1);
    if (power) {
        const int count = mode_powers(N);
        mode_power_kernel<<<(count + 255) / 256, 256, 0, s>>>(power, count, p);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    fill_modes_kernel<<<grid_for(total, sm_count, 8), 256, (N / 4 + 1) * sizeof(double2), s>>>(modes, power, p);
    return cudaGetLastError();
}

cudaError_t launch_assemble(int dtype, void *dst, const double *delta, double base, double scale, int N, long long P,
                            long long PP, cudaStream_t s)
{
    const unsigned grid = (unsigned)(((size_t)N * N * (N / 4) + 255) / 256);
    if (dtype == TL_F32)
        assemble_kernel<float><<<grid, 256, 0, s>>>(static_cast<float *>(dst), delta, base, (float)base, scale, N, P, PP);
    else
        assemble_kernel<double><<<grid, 256, 0, s>>>(static_cast<double *>(dst), delta, base, base, scale, N, P, PP);
    return cudaGetLastError();
}

cudaError_t launch_widen(int dtype, double *dst, const void *src, double *offset, int N, long long P, long long PP,
                         cudaStream_t s)
{
    const unsigned grid = (unsigned)(((size_t)N * N * (N / 4) + 255) / 256);
    if (dtype == TL_F32)
        widen_kernel<float><<<grid, 256, 0, s>>>(dst, static_cast<const float *>(src), offset, N, P, PP);
    else
        widen_kernel<double><<<grid, 256, 0, s>>>(dst, static_cast<const double *>(src), offset, N, P, PP);
    return cudaGetLastError();
}

cudaError_t launch_bin(const double2 *modes, int N, int nbins, double *Psum, double *rsum, unsigned long long *cnt,
                       double *mode0, int sm_count, cudaStream_t s)
{
    const size_t total = (size_t)(N / 2 + 1) * (N / 2 + 2) / 2 * (N / 4 + 1);
    const size_t smem = (size_t)(N / 4 + 1) * sizeof(double2) +
                        (size_t)nbins * (2 * sizeof(double) + sizeof(unsigned long long));
    if (smem > 48 * 1024) {  // N above 1976
        static SmemLimit limit;
        const cudaError_t e = limit.raise(bin_kernel, smem);
        if (e != cudaSuccess) return e;
    }
    bin_kernel<<<grid_for(total, sm_count, 2), 256, smem, s>>>(modes, N, nbins, Psum, rsum, cnt, mode0);
    return cudaGetLastError();
}

}  // namespace tl
