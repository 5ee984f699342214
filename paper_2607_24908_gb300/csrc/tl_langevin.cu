// Langevin evolution of a scalar phi^4 field (the paper's interface example,
// Sec. 2, Eq. 1): Euler-Maruyama steps
//     phi <- phi + dt (Lap phi - m^2 phi - (lambda/2) phi^3) + noise sqrt(dt) xi,
// with xi a unit Gaussian per site and step (the paper's field-valued random
// number generator rescaled by 1/sqrt(dt)).  The sites with dense indices 2k
// and 2k + 1 share one Philox-2x64-10 draw of counter (k, 2^63 + step) under
// key seed; Box-Muller on its two words gives two independent Gaussians, the
// cosine one for site 2k and the sine one for site 2k + 1 (half the generator
// work of one draw per site, which bounds this kernel).
//
// One kernel per step, marching z-planes like the fused pass: phi at z-1, z,
// z+1 in registers, the y-neighbour rows and edge sites through L1/L2; HBM
// sees one read and one write of phi per site.  The field ping-pongs between
// the lattice's two phi_0 buffers; momenta are not used.
#include <math.h>
#include <stdint.h>

#include "tl_boxmuller.cuh"
#include "tl_internal.cuh"
#include "tl_lattice.cuh"
#include "tl_philox.cuh"

namespace {

using tl::philox2x64_10_low;  // the initial-state draw's generator

// The two Gaussians of draw k: (cos, sin) halves of Box-Muller.
__device__ __forceinline__ void gauss2(const tl::BoxMullerTable *t, uint32_t k, uint64_t ctr1, uint64_t seed, double &gc,
                                       double &gs)
{
    uint64_t w0, w1;
    philox2x64_10_low(k, ctr1, seed, w0, w1);
    const double r = sqrt(2.0 * tl::neg_log_u53(t, (w0 >> 11) + 1));
    double s, c;
    tl::unit_circle_u53(t, w1 >> 11, c, s);
    gc = r * c;
    gs = r * s;
}

// x 2^-53 for an integer 0 <= x <= 2^53, formed in FP32 without FP64
// arithmetic (GB300's FP64 pipe is slow): x = hi 2^29 + lo, hi <= 2^24 exact,
// lo < 2^29 rounded once on conversion, one more rounding in the fma; the
// result keeps a relative precision of about 2^-24 at any magnitude, so small
// u1 (the Gaussian tail) stays as accurate as in a correctly rounded FP64->FP32
// conversion.
__device__ __forceinline__ float u53_f32(uint64_t x)
{
    const uint32_t hi = (uint32_t)(x >> 29), lo = (uint32_t)(x & 0x1FFFFFFFu);
    return fmaf((float)hi, 0x1p-24f, (float)lo * 0x1p-53f);
}

// (cos, sin)(2 pi u) in FP32 for u = (w >> 11) 2^-53: the nearest quarter turn
// is taken off in integers, the rest, within an eighth of a turn, goes into the
// Taylor polynomials (first omitted terms below 2e-9 and 3e-8).  The rest enters
// in two parts, 30 bits and the 21 below them (exact in FP32), so that the
// component that vanishes near an axis keeps its relative accuracy however small it
// is.  Half of the instructions are on the FMA pipes; sincospif of a converted
// uniform took 35.
__device__ __forceinline__ void unit_circle(uint64_t w, float &c, float &s)
{
    constexpr float kTurn32 = (float)(2.0 * M_PI / 4294967296.0);
    const uint32_t h = (uint32_t)(w >> 32) + 0x20000000u, low = (uint32_t)w & ~0x7ffu;
    const float x = fmaf((float)low, kTurn32 * 0x1p-32f, (float)((int32_t)(h & 0x3fffffffu) - 0x20000000) * kTurn32);
    const float t = x * x;
    float ps = fmaf(t, 1.0f / 362880.0f, -1.0f / 5040.0f);
    ps = fmaf(ps, t, 1.0f / 120.0f);
    ps = fmaf(ps, t, -1.0f / 6.0f);
    ps = fmaf(ps * t, x, x);
    float pc = fmaf(t, 1.0f / 40320.0f, -1.0f / 720.0f);
    pc = fmaf(pc, t, 1.0f / 24.0f);
    pc = fmaf(pc, t, -0.5f);
    pc = fmaf(pc, t, 1.0f);
    const bool odd = h & 0x40000000u;  // quarter turns 0..3 in the top two bits
    const uint32_t u = __float_as_uint(odd ? ps : pc), v = __float_as_uint(odd ? pc : ps);
    c = __uint_as_float(u ^ ((h ^ (h << 1)) & 0x80000000u));  // cos is negative in quarters 1, 2
    s = __uint_as_float(v ^ (h & 0x80000000u));               // sin in 2, 3
}

__device__ __forceinline__ void gauss2(const tl::BoxMullerTable *, uint32_t k, uint64_t ctr1, uint64_t seed, float &gc,
                                       float &gs)
{
    uint64_t w0, w1;
    philox2x64_10_low(k, ctr1, seed, w0, w1);
    // Box-Muller in FP32 (the field is stored in FP32): u1 to 2^-24 of itself,
    // the angle to 2^-23 of its distance from the nearest axis
    const float u1 = u53_f32((w0 >> 11) + 1);
    const float r = sqrtf(-2.0f * logf(u1));
    float s, c;
    unit_circle(w1, c, s);
    gc = r * c;
    gs = r * s;
}

// W consecutive sites (one 16-byte word: rows start on 128-byte boundaries).
__device__ __forceinline__ void ld(const float *p, float (&o)[4])
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w;
}
__device__ __forceinline__ void ld(const double *p, double (&o)[2])
{
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    o[0] = v.x, o[1] = v.y;
}
__device__ __forceinline__ void st(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st(double *p, const double (&v)[2])
{
    *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
}

// FP32 is bound by instruction issue and the integer pipes (the draws' wide
// products alone take 150 us at 384^3): neighbours come as 16-byte words and by
// shuffle, the angle from the word's bits, the first round of the generator
// with two products; 467 instructions a plane and thread, from 538, and less
// in the last wave: 303 -> 244 us at 384^3, of which the angle's second part took
// back 4 (248).  FP64 is bound by the FP64 pipe: the
// table form of Box-Muller (tl_boxmuller.cuh) took 384^3 from 5910 to 3951 us.
template <typename T>
__global__ void __launch_bounds__(256) langevin_pass(const T *__restrict__ in, T *__restrict__ out, int N, int txt,
                                                     int ty, int zc, long long P, long long PP, T inv_dx2, T dt, T m2,
                                                     T half_lam, T amp, uint64_t seed, uint64_t ctr1)
{
    constexpr int W = 16 / (int)sizeof(T);
    constexpr bool kTable = sizeof(T) == 8;
    __shared__ __align__(16) unsigned char table_raw[kTable ? sizeof(tl::BoxMullerTable) : 16];
    tl::BoxMullerTable *table = reinterpret_cast<tl::BoxMullerTable *>(table_raw);
    if (kTable) tl::load_box_muller(table);
    const int tx = threadIdx.x % txt, tyi = threadIdx.x / txt;
    const int x0 = (blockIdx.x * txt + tx) * W;
    const int y = blockIdx.y * ty + tyi;
    const int z0 = blockIdx.z * zc;
    const int z1 = min(z0 + zc, N);
    const bool active = tyi < ty && x0 < N && y < N;
    // the x-neighbours are in the adjacent lanes' words; a thread at a row end,
    // a tile edge or a warp edge loads its own.  The mask of the shuffles is formed
    // while the warp is whole: every lane that stays is in it
    const unsigned lanes = __ballot_sync(0xffffffffu, active);
    if (!active) return;
    const int lane = threadIdx.x & 31;
    const bool own_l = tx == 0 || lane == 0, own_r = tx == txt - 1 || x0 + W == N || lane == 31;
    const int src_l = own_l ? lane : lane - 1, src_r = own_r ? lane : lane + 1;
    const size_t row = (size_t)y * P + x0;
    const T *pc = in + (size_t)z0 * PP + row;  // this thread's sites of plane z
    T *po = out + (size_t)z0 * PP + row;
    const long long dym = (y == 0 ? N - 1 : -1) * P, dyp = (y + 1 == N ? 1 - N : 1) * P;
    const int dxl = x0 == 0 ? N - 1 : -1, dxr = x0 + W == N ? W - N : W;
    const long long up = (1 - (long long)N) * PP;  // from plane N - 1 to plane 0
    // ghost rows of this thread's sites (padded arrays carry one ghost row on
    // each side of a plane; the x-edges need no copies)
    const long long gy = y == 0 ? (long long)N * P : (y == N - 1 ? -(long long)N * P : 0);
    // x0 and W are even: the thread's sites form whole pairs; N <= 2048: pair indices are below 2^32
    uint32_t k0 = (uint32_t)((((uint64_t)z0 * N + y) * N + x0) >> 1);
    const uint32_t dk = (uint32_t)N * N / 2;
    T zm[W], cu[W], zp[W];
    ld(z0 == 0 ? pc - up : pc - PP, zm);
    ld(pc, cu);
    for (int z = z0; z < z1; ++z) {
        T ym[W], yp[W];
        ld(z + 1 == N ? pc + up : pc + PP, zp);
        ld(pc + dym, ym);
        ld(pc + dyp, yp);
        T a = __shfl_sync(lanes, cu[W - 1], src_l), b = __shfl_sync(lanes, cu[0], src_r);
        if (own_l) a = __ldg(pc + dxl);
        if (own_r) b = __ldg(pc + dxr);
        T xi[W];
#pragma unroll
        for (int j = 0; j < W; j += 2) gauss2(table, k0 + j / 2, ctr1, seed, xi[j], xi[j + 1]);
        T o[W];
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const T c = cu[j];
            const T left = j == 0 ? a : cu[j - 1];
            const T right = j == W - 1 ? b : cu[j + 1];
            const T lap = (((left - c) + (right - c)) + ((ym[j] - c) + (yp[j] - c))) + ((zm[j] - c) + (zp[j] - c));
            const T drift = lap * inv_dx2 - m2 * c - half_lam * c * c * c;
            o[j] = (c + dt * drift) + amp * xi[j];
        }
        st(po, o);
        if (gy) st(po + gy, o);
#pragma unroll
        for (int j = 0; j < W; ++j) {
            zm[j] = cu[j];
            cu[j] = zp[j];
        }
        pc += PP;
        po += PP;
        k0 += dk;
    }
}

}  // namespace

extern "C" int tl_langevin_step(tl_lattice *L, int n, double dt, const tl_langevin_params *p, uint64_t seed)
{
    tl::NvtxScope nvtx_range("tl_langevin_step");
    tl::set_error(TL_OK, "", "");
    if (!L || !p) return tl::fail(TL_EINVAL, "NULL argument");
    if (n < 0 || !(dt > 0.0) || !isfinite(dt)) return tl::fail(TL_EINVAL, "n >= 0 and a positive finite dt needed");
    if (!isfinite(p->lambda) || !isfinite(p->m2) || !isfinite(p->noise)) return tl::fail(TL_EINVAL, "non-finite parameter");
    if (!(L->state_mask & 1u)) return tl::fail(TL_ESTATE, "phi_0 has not been set");
    if (L->batch_refs > 0) return tl::fail(TL_ESTATE, "lattice is part of a batch");
    tl::PassTuning t{tl::kVariantLdg, 8, 0, L->N, 0, 256, 0};
    tl::PassGeom g = tl::pass_geometry(L->N, (int)L->esz, L->sm_count, 1, t);
    int per_sm = 0;
    cudaError_t oe = L->dtype == TL_F32
                         ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, langevin_pass<float>, 256, 0)
                         : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, langevin_pass<double>, 256, 0);
    if (oe != cudaSuccess) return tl::fail(TL_ECUDA, "langevin occupancy: %s", cudaGetErrorString(oe));
    // z-chunk.  FP64 is bound by arithmetic alone, which the two planes a chunk
    // reads beyond its own do not add to: one plane per CTA spreads it best (us, with two
    // operations a draw less than now:
    // 100^3 96 against 116 with 4 planes, 212^3 777 against 795, 384^3 3779 against
    // 3790).  FP32: the fewest (waves of CTAs) x (planes per CTA + 1/4 for those two
    // planes; measured before the angle had its second part): 384^3 244 us with 19
    // planes, 258 with 32; 64^3 5.7 with 1, 6.8 with 4.
    const long slots = (long)(L->sm_count > 0 ? L->sm_count : 152) * (per_sm > 0 ? per_sm : 1);
    double best = 0.0;
    for (int c = 1; c <= (L->dtype == TL_F32 ? L->N : 1); ++c) {
        const long ctas = (long)g.grid.x * g.grid.y * ((L->N + c - 1) / c);
        const double cost = (double)((ctas + slots - 1) / slots) * (c + 0.25);
        if (best == 0.0 || cost < best) best = cost, g.zc = c;
    }
    g.grid.z = (unsigned)((L->N + g.zc - 1) / g.zc);
    const double inv_dx2 = 1.0 / (L->dx * L->dx);
    const double amp = p->noise * sqrt(dt);
    for (int s = 0; s < n; ++s) {
        void *in = L->buf[L->cur][0][0];
        void *out = L->buf[L->cur ^ 1][0][0];
        const uint64_t ctr1 = (1ull << 63) + (uint64_t)(L->langevin_steps + s);
        if (L->dtype == TL_F32)
            langevin_pass<float><<<g.grid, 256, 0, L->stream>>>(
                static_cast<const float *>(in), static_cast<float *>(out), L->N, g.txt, g.ty, g.zc, L->model.pitch,
                L->model.pplane, (float)inv_dx2,
                (float)dt, (float)p->m2, (float)(0.5 * p->lambda), (float)amp, seed, ctr1);
        else
            langevin_pass<double><<<g.grid, 256, 0, L->stream>>>(
                static_cast<const double *>(in), static_cast<double *>(out), L->N, g.txt, g.ty, g.zc, L->model.pitch,
                L->model.pplane, inv_dx2, dt,
                p->m2, 0.5 * p->lambda, amp, seed, ctr1);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return tl::fail(TL_ECUDA, "langevin_pass: %s", cudaGetErrorString(e));
        // phi_0 ping-pongs; the momenta stay where they are
        L->buf[L->cur][0][0] = out;
        L->buf[L->cur ^ 1][0][0] = in;
    }
    L->langevin_steps += n;
    L->energies_valid = false;
    if (n & 1) tl::invalidate_launches(L);  // phi_0's buffers traded places: tensor maps and graphs are stale
    return TL_OK;
}
