// Classical SU(2) Yang-Mills in temporal gauge: the paper's benchmark
// workload (Sec. 4), each step a kick of the electric fields by the plaquette
// staples and a drift of the links by the closed-form SU(2) exponential map.
//
// Links are unit quaternions U = u0 + i u.s, stored on the device as
// quaternion records [direction][site][4] (one 16-byte load per link in FP32,
// two in FP64; consecutive threads read consecutive records); electric fields
// su(2) vectors E = i e.s, component-major [direction][component][site] (only
// a site's own fields are read).  The host layout of both is component-major;
// tl_su2_set_state / tl_su2_get_state transpose the links through the spare
// link buffer.
// One fused pass per step: e_i(x) <- e_i(x) - 2 dt sum_{j != i} Im[U_i S_ij]
// with the old links, then U_i(x) <- exp(dt E_i(x)) U_i(x) written to the
// other link buffer (ping-pong), so the neighbours' staples always see the old
// links.  HBM per site and step: read 12 link + 9 field values, write 9 + 12.
// A separate measurement kernel reduces the electric and plaquette energies
// and the Gauss-law violation in a fixed order (per-CTA slots, one summing CTA).
#include <math.h>
#include <stdint.h>

#include <new>

#include "tl_internal.cuh"
#include "tl_lattice.cuh"
#include "tl_philox.cuh"
#include "tl_smem.cuh"

namespace {

template <typename T>
struct Q {
    T w, x, y, z;
};

__device__ __forceinline__ float fma_su(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_su(double a, double b, double c) { return fma(a, b, c); }

// One multiplication and three fused multiply-adds a component (16 operations;
// left to the compiler's contraction the vector components take five).
template <typename T>
__device__ __forceinline__ Q<T> qmul(const Q<T> &a, const Q<T> &b)
{
    // (a0 + i a.s)(b0 + i b.s) = a0 b0 - a.b + i (a0 b + b0 a - a x b).s
    Q<T> r;
    r.w = fma_su(a.w, b.w, -fma_su(a.x, b.x, fma_su(a.y, b.y, a.z * b.z)));
    r.x = fma_su(a.w, b.x, fma_su(b.w, a.x, fma_su(-a.y, b.z, a.z * b.y)));
    r.y = fma_su(a.w, b.y, fma_su(b.w, a.y, fma_su(-a.z, b.x, a.x * b.z)));
    r.z = fma_su(a.w, b.z, fma_su(b.w, a.z, fma_su(-a.x, b.y, a.y * b.x)));
    return r;
}
template <typename T>
__device__ __forceinline__ Q<T> qadj(const Q<T> &a)
{
    return Q<T>{a.w, -a.x, -a.y, -a.z};
}
// Link record of direction i at site s (records are 16- or 32-byte aligned).
__device__ __forceinline__ Q<float> ldU(const float *U, size_t n3, int i, size_t s)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(U + ((size_t)i * n3 + s) * 4));
    return Q<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Q<double> ldU(const double *U, size_t n3, int i, size_t s)
{
    const double2 *b = reinterpret_cast<const double2 *>(U + ((size_t)i * n3 + s) * 4);
    const double2 a = __ldg(b), c = __ldg(b + 1);
    return Q<double>{a.x, a.y, c.x, c.y};
}
__device__ __forceinline__ void stU(float *U, size_t n3, int i, size_t s, const Q<float> &q)
{
    *reinterpret_cast<float4 *>(U + ((size_t)i * n3 + s) * 4) = make_float4(q.w, q.x, q.y, q.z);
}
__device__ __forceinline__ void stU(double *U, size_t n3, int i, size_t s, const Q<double> &q)
{
    double2 *b = reinterpret_cast<double2 *>(U + ((size_t)i * n3 + s) * 4);
    b[0] = make_double2(q.w, q.x);
    b[1] = make_double2(q.y, q.z);
}

template <typename T>
__device__ __forceinline__ void sincos_t(T a, T *s, T *c);
template <>
__device__ __forceinline__ void sincos_t<float>(float a, float *s, float *c) { sincosf(a, s, c); }
template <>
__device__ __forceinline__ void sincos_t<double>(double a, double *s, double *c) { sincos(a, s, c); }

// The rotation of the drift, exp(i dt e.s) = cos(theta) + i f e.s with
// theta = dt |e| and f = sin(theta) / |e| = dt sin(theta) / theta, from
// q2 = |e|^2.  Small angles (theta^2 below kSmallTheta2, the common case: the
// per-step angle is tiny) use the Taylor series of sin(theta)/theta and
// cos(theta) in theta^2, truncated where the first omitted term is below half
// an ulp of the result (FP32: theta < 1/2, terms to theta^8, first omitted
// term < 3e-10; FP64: theta < 1/4, terms to theta^10 / theta^12, < 1e-17): no
// square root, no division, no trigonometric call.  Larger angles take
// sincos of theta.
template <typename T>
constexpr T kSmallTheta2 = sizeof(T) == 4 ? (T)0.25 : (T)0.0625;

template <typename T>
__device__ __forceinline__ void drift_rotation(T q2, T dt, T *f, T *cs)
{
    const T t2 = dt * dt * q2;
    if (t2 < kSmallTheta2<T>) {
        T sc, cc;
        if (sizeof(T) == 4) {
            // sin(t)/t = sum_k (-t^2)^k / (2k+1)!,  cos(t) = sum_k (-t^2)^k / (2k)!
            sc = (T)(1.0 / 362880.0);
            sc = sc * t2 - (T)(1.0 / 5040.0);
            sc = sc * t2 + (T)(1.0 / 120.0);
            sc = sc * t2 - (T)(1.0 / 6.0);
            cc = (T)(1.0 / 40320.0);
            cc = cc * t2 - (T)(1.0 / 720.0);
            cc = cc * t2 + (T)(1.0 / 24.0);
            cc = cc * t2 - (T)(1.0 / 2.0);
        } else {
            sc = (T)(-1.0 / 39916800.0);
            sc = sc * t2 + (T)(1.0 / 362880.0);
            sc = sc * t2 - (T)(1.0 / 5040.0);
            sc = sc * t2 + (T)(1.0 / 120.0);
            sc = sc * t2 - (T)(1.0 / 6.0);
            cc = (T)(1.0 / 479001600.0);
            cc = cc * t2 - (T)(1.0 / 3628800.0);
            cc = cc * t2 + (T)(1.0 / 40320.0);
            cc = cc * t2 - (T)(1.0 / 720.0);
            cc = cc * t2 + (T)(1.0 / 24.0);
            cc = cc * t2 - (T)(1.0 / 2.0);
        }
        *f = dt * (sc * t2 + (T)1);
        *cs = cc * t2 + (T)1;
    } else {
        const T nrm = sqrt(q2);
        T sn;
        sincos_t<T>(dt * nrm, &sn, cs);
        *f = sn / nrm;
    }
}

template <typename T>
struct alignas(4 * sizeof(T)) Rec {
    T w, x, y, z;
};

// F += sg (V - R(W^+) v) (FIRST: F = that), with R(W^+) v = Im(W^+ (0, v) W)
// the vector v rotated by the adjoint action of W^+.  For W = w + i u.s,
//   R(W^+) v = (w^2 - |u|^2) v + 2 (u.v) u + 2 w (u x v),
// which for a unit W is v + w c + u x c with c = 2 u x v; that form is
// accumulated here, term by term (21 operations and the 3 of 2 u, which the two
// forces a link rotates for share; with the factors on the products it took
// 25).  Links are unit quaternions anyway: the plaquette form of the backward
// staple itself uses W^+ W = 1.
template <bool FIRST, typename T>
__device__ __forceinline__ void add_force(const Q<T> &W, const Rec<T> &V, const Rec<T> &v, T sg, T &Fx, T &Fy, T &Fz)
{
    const T ux = (T)2 * W.x, uy = (T)2 * W.y, uz = (T)2 * W.z;
    const T cx = fma_su(uy, v.z, -(uz * v.y)), cy = fma_su(uz, v.x, -(ux * v.z)), cz = fma_su(ux, v.y, -(uy * v.x));
    const T w = -sg * W.w, x = -sg * W.x, y = -sg * W.y, z = -sg * W.z;  // signs of the operands
    const T ax = FIRST ? sg * V.x : Fx + sg * V.x, ay = FIRST ? sg * V.y : Fy + sg * V.y,
            az = FIRST ? sg * V.z : Fz + sg * V.z;
    Fx = fma_su(y, cz, fma_su(-z, cy, fma_su(w, cx, ax - sg * v.x)));
    Fy = fma_su(z, cx, fma_su(-x, cz, fma_su(w, cy, ay - sg * v.y)));
    Fz = fma_su(x, cy, fma_su(-y, cx, fma_su(w, cz, az - sg * v.z)));
}

// One pass per step over CTAs of tx x ty site columns (Su2Tile), each marching
// z-planes.  The force on U_i(x) is Im[U_i(x) S_i(x)] with the staples S of
// Sec. 4; in terms of the plaquettes
//   P_ij(x) = U_i(x) U_j(x+i) U_i(x+j)^+ U_j(x)^+,   V_ij = Im P_ij = -V_ji,
// U_i f_ij(x) = P_ij(x) and, for unit links, U_i b_ij(x) = W^+ P_ij(x-j)^+ W
// with W = U_j(x-j), so
//   Im[U_i S_i](x) = sum_{j != i} V_ij(x) - R(W^+) V_ij(x-j),
// R(W^+) the rotation of add_force.  Each plaquette is then formed once per site
// (three per site, instead of four staples per link) and shared through shared
// memory: V_xy, V_xz, V_yz of the CTA's tile plus the -x / -y halo it needs,
// in two buffers (plane z, and z+1 being formed); the plaquettes of plane z-1
// are needed only at a thread's own site and stay in its registers.
//
// The link records of a plane's tile with a one-site halo, (ty + 2) x (tx + 2)
// sites x 3 directions, are copied into a ring of shared-memory stages with
// cp.async (16-byte chunks, addresses wrapped periodically by the copying
// thread) one plane ahead of their first use.  Stage s holds the plane with
// relative index (z - z0 + 1) % 4 == s.
constexpr int kSu2Stages = 4;
constexpr int kSu2PlaqBufs = 2;      // planes z (read) and z+1 (written)
constexpr int kSu2MaxHalo = 340;     // (tx + 2) (ty + 2): the records a thread's copy slots cover
constexpr int kSu2MaxPlaq = 297;     // (tx + 1) (ty + 1)

// Tile shape and division of the lattice's site columns (tiles x N planes)
// among the CTAs.
struct Su2Tile {
    int tx, ty;    // tile of site columns, tx ty <= 256 threads
    int ntx, nty;  // tiles along x and y
    int zc;        // planes per CTA, CTAs in z-chunk-major order; 0: even division (see su2_tile)
};

constexpr size_t su2_smem(int tx, int ty, size_t esz, bool stage_fields)
{
    return (size_t)(kSu2Stages * 3 * (tx + 2) * (ty + 2) + kSu2PlaqBufs * 3 * (tx + 1) * (ty + 1)) * 4 * esz +
           (stage_fields ? 2 * 9 * 256 * esz : 0);  // two planes of electric fields
}

__device__ __forceinline__ void cp_async_cg16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// FIXED: a 32 x 8 tile with compile-time strides.  STAGE: the electric fields
// come through shared memory (cp.async, each thread its own nine values) one
// plane ahead, instead of through registers.
//
// FP64 is bound by the FP64 pipe (438 of its issue slots a site at 192^3, from
// 576); what counts is that no lane, CTA slot or operation is wasted (see
// su2_plan).  FP32 issues about 740 warp instructions per 32 sites,
// half of them addresses, shared-memory traffic and copies, on 57% of the cycles
// at 16 warps per SM, and moves its bytes at 0.56 (128^3) to 0.78 (256^3) of
// the measured HBM rate.
// us per step, before -> now (before: 32 x 8 tiles and equal z-chunks for
// every N, products of five operations a component, three plaquette buffers):
//   FP64  33^3 114 -> 53   64^3 283 -> 209   100^3 1383 -> 759   128^3 1959 -> 1486   192^3 6513 -> 4950
//   FP32  33^3 10.3 -> 8.4   100^3 57.6 -> 51   128^3 84.4 -> 76.3   150^3 145 -> 132   192^3 248 -> 231   256^3 568 -> 532
template <typename T, bool FIXED, bool STAGE>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1)
    su2_pass(const T *__restrict__ U, T *__restrict__ Uout, T *__restrict__ E, int N, Su2Tile tile, T dt)
{
    extern __shared__ __align__(16) unsigned char su2_raw[];
    const int Tx = FIXED ? 32 : tile.tx, Ty = FIXED ? 8 : tile.ty;
    const int Hx = Tx + 2, Hxy = (Tx + 2) * (Ty + 2), stage_recs = 3 * Hxy;  // link tile with its one-site halo
    const int Px = Tx + 1, Pxy = (Tx + 1) * (Ty + 1), plaq_recs = 3 * Pxy;   // plaquette tile with the -x / -y halo
    Rec<T> *ring = reinterpret_cast<Rec<T> *>(su2_raw);
    Rec<T> *plaq = ring + kSu2Stages * stage_recs;
    const int tid = threadIdx.x;
    const int ty = tid / Tx, tx = tid - ty * Tx;
    const size_t n3 = (size_t)N * N * N;
    const size_t NN = (size_t)N * N;
    const int rx = tx + 1, ry = ty + 1;
    const int own = ry * Hx + rx;    // this thread's site in a link tile
    const int pown = ry * Px + rx;   // and in a plaquette tile

    // this CTA's planes, counted through the tiles: [p, pend)
    const int tiles = tile.ntx * tile.nty;
    int p, pend;
    if (tile.zc > 0) {
        const int t = blockIdx.x % tiles, z = blockIdx.x / tiles * tile.zc;
        p = t * N + z;
        pend = t * N + min(z + tile.zc, N);
    } else {
        p = (int)((long long)blockIdx.x * tiles * N / gridDim.x);
        pend = (int)((long long)(blockIdx.x + 1) * tiles * N / gridDim.x);
    }

    while (p < pend) {  // one tile's planes z0 .. z1 - 1 at a time
        const int t = p / N, z0 = p - t * N, z1 = min(N, z0 + (pend - p));
        p += z1 - z0;
        const int x0 = t % tile.ntx * Tx, y0 = t / tile.ntx * Ty;
        const int x = x0 + tx, y = y0 + ty;
        const bool active = ty < Ty && x < N && y < N;

        // this thread's copy chunks: chunk r of a stage is half (r % C) of record
        // r / C = (i * Hy + ry) * Hx + rx; its source packed as wx | wy << 11 |
        // i << 22 | half << 24 (N <= 1290 < 2^11)
        constexpr int C = (int)sizeof(T) / 4;
        constexpr int kSlots = (3 * kSu2MaxHalo * C + 255) / 256;
        const int chunks = stage_recs * C;
        unsigned src[kSlots];
#pragma unroll
        for (int k = 0; k < kSlots; ++k) {
            const int r = tid + 256 * k;
            const int rec = r / C, half = r % C;
            const int i = rec / Hxy, q = rec - i * Hxy, qy = q / Hx;
            const int wx = (x0 - 1 + (q - qy * Hx) + N) % N, wy = (y0 - 1 + qy + N) % N;
            src[k] = (unsigned)wx | (unsigned)wy << 11 | (unsigned)(i & 3) << 22 | (unsigned)half << 24;
        }
        auto copy_plane = [&](int z) {
            const int zz = z < 0 ? z + N : (z >= N ? z - N : z);
            unsigned char *st =
                reinterpret_cast<unsigned char *>(ring + ((z - z0 + 1) & (kSu2Stages - 1)) * stage_recs);
            const T *Uz = U + (size_t)zz * NN * 4;
#pragma unroll
            for (int k = 0; k < kSlots; ++k) {
                const int r = tid + 256 * k;
                const unsigned v = src[k];
                const size_t rec = (size_t)((v >> 22) & 3u) * n3 + (size_t)((v >> 11) & 2047u) * N + (v & 2047u);
                if (r < chunks) cp_async_cg16(st + (size_t)r * 16, Uz + rec * 4 + (v >> 24) * (16 / sizeof(T)));
            }
            cp_async_commit();
        };
        // link i at tile site `at` of the plane with relative index zr = z - z0 + 1
        auto link = [&](int i, int at, int zr) -> Q<T> {
            const Rec<T> v = ring[(zr & (kSu2Stages - 1)) * stage_recs + i * Hxy + at];
            return Q<T>{v.w, v.x, v.y, v.z};
        };
        // V_ij at tile site `at` of plane zr (i < j; reads planes zr and zr + 1)
        auto plaq_im = [&](int i, int j, int at, int zr) -> Rec<T> {
            const Q<T> a = link(i, at, zr);
            const Q<T> b = link(j, at + (i == 0 ? 1 : Hx), zr);  // x + i, i = x or y
            const Q<T> c = link(i, at + (j == 1 ? Hx : 0), zr + (j == 2));
            const Q<T> d = link(j, at, zr);
            const Q<T> q = qmul(qmul(a, b), qadj(qmul(d, c)));
            return Rec<T>{(T)0, q.x, q.y, q.z};
        };
        // the halo plaquette of thread tid < 2 (Tx + Ty): row y0-1 (V_xy, V_yz),
        // column x0-1 (V_xy, V_xz), the pair (i, j) as data so that the warp stays together
        const bool hrow = tid < 2 * Tx;
        const int hs = hrow ? (tid < Tx ? tid : tid - Tx) : (tid < 2 * Tx + Ty ? tid - 2 * Tx : tid - 2 * Tx - Ty);
        const int hi = hrow && tid >= Tx ? 1 : 0;
        const int hj = hrow ? (tid < Tx ? 1 : 2) : (tid < 2 * Tx + Ty ? 1 : 2);
        const int hx = hrow ? 1 + hs : 0, hy = hrow ? 0 : 1 + hs;
        const bool halo = tid < 2 * (Tx + Ty) && x0 + hx <= N && y0 + hy <= N;
        // plaquettes of plane zr into buffer zr & 1 (and this site's into V)
        auto form_plaquettes = [&](int zr, Rec<T>(&V)[3]) {
            Rec<T> *b = plaq + (zr & 1) * plaq_recs;
            if (active) {
                V[0] = plaq_im(0, 1, own, zr);
                V[1] = plaq_im(0, 2, own, zr);
                V[2] = plaq_im(1, 2, own, zr);
#pragma unroll
                for (int k = 0; k < 3; ++k) b[k * Pxy + pown] = V[k];
            }
            if (halo) b[(hi + hj - 1) * Pxy + hy * Px + hx] = plaq_im(hi, hj, hy * Hx + hx, zr);
        };

        // Software pipeline, one barrier per plane: the interval of plane z forms
        // the plaquettes of plane z+1 and then updates the links of plane z from
        // the plaquettes of planes z and z-1 (formed in earlier intervals).  Ring
        // stages hold planes z..z+2 while z+3 lands; U_z(x - z) is carried in
        // registers from the previous plane, whose stage is being refilled.
        copy_plane(z0 - 1);
        copy_plane(z0);
        copy_plane(z0 + 1);
        copy_plane(z0 + 2);
        cp_async_wait_all();
        __syncthreads();
        Q<T> uz_prev{0, 0, 0, 0};
        Rec<T> Vz[2], V[3];  // V_xz, V_yz of plane z - 1; V_xy, V_xz, V_yz of plane z
        if (active) {        // plane z0 - 1 (relative index 0) for the first plane's -z terms
            Vz[0] = plaq_im(0, 2, own, 0);
            Vz[1] = plaq_im(1, 2, own, 0);
            uz_prev = link(2, own, 0);
        }
        form_plaquettes(1, V);
        // the electric fields of a plane are loaded one plane ahead of their update
        T eo[9], en[9];
        T *es = reinterpret_cast<T *>(plaq + kSu2PlaqBufs * plaq_recs) + tid;
        const size_t s0 = (size_t)z0 * NN + (size_t)y * N + x;
        auto copy_fields = [&](int z, size_t s) {
#pragma unroll
            for (int c = 0; c < 9; ++c) cp_async_4(es + (((z & 1) * 9 + c) << 8), E + (size_t)c * n3 + s);
        };
        if (active) {
            if constexpr (STAGE) {
                copy_fields(z0, s0);
            } else {
#pragma unroll
                for (int c = 0; c < 9; ++c) eo[c] = E[(size_t)c * n3 + s0];
            }
        }
        for (int z = z0; z < z1; ++z) {
            const int zr = z - z0 + 1;
            const Rec<T> *cur = plaq + (zr & 1) * plaq_recs;
            cp_async_wait_all();
            __syncthreads();  // plaquettes of plane z complete, plane z+2 landed; the stage of z-1 and the other buffer are free
            if (z + 3 <= z1) copy_plane(z + 3);
            const size_t s = (size_t)z * NN + (size_t)y * N + x;
            if (active && z + 1 < z1) {
                if constexpr (STAGE) {
                    copy_fields(z + 1, s + NN);
                } else {
#pragma unroll
                    for (int c = 0; c < 9; ++c) en[c] = E[(size_t)c * n3 + s + NN];
                }
            }
            Rec<T> Vn[3];
            if (z + 1 < z1) form_plaquettes(zr + 1, Vn);
            if (!active) continue;
            const Q<T> uz = link(2, own, zr);
            if constexpr (STAGE) {
#pragma unroll
                for (int c = 0; c < 9; ++c) eo[c] = es[((z & 1) * 9 + c) << 8];
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                T Fx, Fy, Fz;
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    if (j == i) continue;
                    const int k = i + j - 1;  // (0,1) -> 0, (0,2) -> 1, (1,2) -> 2
                    const T sg = i < j ? (T)1 : (T)-1;
                    // V_ij(x - j) and W = U_j(x - j)
                    const Rec<T> vn = j == 0 ? cur[k * Pxy + pown - 1] : j == 1 ? cur[k * Pxy + pown - Px] : Vz[i];
                    const Q<T> W = j == 0 ? link(0, own - 1, zr) : j == 1 ? link(1, own - Hx, zr) : uz_prev;
                    if (j == (i == 0 ? 1 : 0)) add_force<true>(W, V[k], vn, sg, Fx, Fy, Fz);
                    else add_force<false>(W, V[k], vn, sg, Fx, Fy, Fz);
                }
                const T e1 = eo[3 * i] - (T)2 * dt * Fx;
                const T e2 = eo[3 * i + 1] - (T)2 * dt * Fy;
                const T e3 = eo[3 * i + 2] - (T)2 * dt * Fz;
                T *ei = E + (size_t)(3 * i) * n3 + s;
                ei[0] = e1;
                ei[n3] = e2;
                ei[2 * n3] = e3;
                // drift: exp(i dt e.s) = cos(dt|e|) + i sin(dt|e|) e/|e|
                T f, cs;
                drift_rotation<T>(e1 * e1 + e2 * e2 + e3 * e3, dt, &f, &cs);
                Q<T> u = qmul(Q<T>{cs, f * e1, f * e2, f * e3}, i == 2 ? uz : link(i, own, zr));
                if (sizeof(T) == 4) {  // FP32 storage: keep the link on the unit sphere
                    const T r = rsqrt(u.w * u.w + u.x * u.x + u.y * u.y + u.z * u.z);
                    u = Q<T>{u.w * r, u.x * r, u.y * r, u.z * r};
                }
                stU(Uout, n3, i, s, u);
            }
            uz_prev = uz;
            Vz[0] = V[1];
            Vz[1] = V[2];
#pragma unroll
            for (int k = 0; k < 3; ++k) V[k] = Vn[k];
            if constexpr (!STAGE) {
#pragma unroll
                for (int c = 0; c < 9; ++c) eo[c] = en[c];
            }
        }
        cp_async_wait_all();
        __syncthreads();  // the ring and the plaquette buffers are the next tile's
    }
}

// A stored value in FP64.  INT forms a float's double from its bits (exponent
// rebiased, mantissa moved) with integer instructions: a conversion
// instruction runs at the rate of the FP64 pipe, which bounds su2_measure.
// That holds for zeros and normal values; odd_value marks the others.
template <bool INT>
__device__ __forceinline__ double widen(double v)
{
    return v;
}
template <bool INT>
__device__ __forceinline__ double widen(float v)
{
    if constexpr (!INT) return (double)v;
    const unsigned b = __float_as_uint(v), m = b & 0x7fffffffu;
    const unsigned hi = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(b << 29));
}
template <bool INT, typename T>
__device__ __forceinline__ Q<double> widen(const Q<T> &q)
{
    return Q<double>{widen<INT>(q.w), widen<INT>(q.x), widen<INT>(q.y), widen<INT>(q.z)};
}
__device__ __forceinline__ bool odd_value(double) { return false; }
__device__ __forceinline__ bool odd_value(float v)  // subnormal, infinite or NaN
{
    const unsigned m = __float_as_uint(v) & 0x7fffffffu;
    return m - 1u < 0x7fffffu || m >= 0x7f800000u;
}

// One site's stored values: its links and fields, the links at x + d, the
// links and fields at x - d.
template <typename T>
struct Su2Site {
    Q<T> c[3], p[6], m[3];  // p: U_j(x+i), U_i(x+j) of the pairs (x,y), (x,z), (y,z)
    T e[9], em[9];
    __device__ __forceinline__ bool odd() const
    {
        if (sizeof(T) == 8) return false;
        bool o = false;
        auto quat = [&](const Q<T> &q) { o |= odd_value(q.w) | odd_value(q.x) | odd_value(q.y) | odd_value(q.z); };
#pragma unroll
        for (int k = 0; k < 3; ++k) quat(c[k]), quat(m[k]);
#pragma unroll
        for (int k = 0; k < 6; ++k) quat(p[k]);
#pragma unroll
        for (int k = 0; k < 9; ++k) o |= odd_value(e[k]) | odd_value(em[k]);
        return o;
    }
    // Adds the site's |e|^2 and 1 - Re P_ij, returns |G|^2.
    template <bool INT>
    __device__ __forceinline__ double add(double &el, double &mag) const
    {
        Q<double> u[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = widen<INT>(c[i]);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i + 1; j < 3; ++j) {
                const Q<double> A = qmul(u[i], widen<INT>(p[2 * (i + j - 1)]));
                const Q<double> B = qmul(u[j], widen<INT>(p[2 * (i + j - 1) + 1]));
                mag += 1.0 - (A.w * B.w + (A.x * B.x + A.y * B.y + A.z * B.z));
            }
        double G[3] = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double ax = widen<INT>(e[3 * i]), ay = widen<INT>(e[3 * i + 1]), az = widen<INT>(e[3 * i + 2]);
            el += ax * ax + ay * ay + az * az;
            // Gauss: E_i(x) - R(W^+) v with W = U_i(x-i), v = E_i(x-i)
            const Q<double> W = widen<INT>(m[i]);
            const double vx = widen<INT>(em[3 * i]), vy = widen<INT>(em[3 * i + 1]), vz = widen<INT>(em[3 * i + 2]);
            const double k = W.w * W.w - (W.x * W.x + W.y * W.y + W.z * W.z);
            const double d = 2.0 * (W.x * vx + W.y * vy + W.z * vz), w2 = 2.0 * W.w;
            const double cx = W.y * vz - W.z * vy, cy = W.z * vx - W.x * vz, cz = W.x * vy - W.y * vx;
            G[0] += ax - fma(w2, cx, fma(d, W.x, k * vx));
            G[1] += ay - fma(w2, cy, fma(d, W.y, k * vy));
            G[2] += az - fma(w2, cz, fma(d, W.z, k * vz));
        }
        return G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
    }
};

// Per-CTA partial sums of |e|^2, 1 - Re P_ij and |G|^2, and the CTA's max
// |G|^2, into slots[4 * cta + q].
//
// Bound by the FP64 pipe (links and fields are read a few times each from
// L1/L2).  Per site, in FP64 operations: Re P_ij = Re[(U_i U_j(x+i)) (U_j
// U_i(x+j))^+] is two products and a four-term dot product (36 instead of the
// 48 of three products), Gauss's term is the rotation formula of add_force in
// its general form, valid for links of any norm (26 instead of two products),
// FP32 values are widened by integer instructions (66 conversions less), the
// square root of |G| is taken once per lattice, on the largest |G|^2, and the
// factors 1/2 and 2 once per lattice.  219 operations a site, the pipe 92% busy:
// FP32 128^3 1386 -> 821 us, FP64 100^3 530 -> 395 us.
template <typename T>
__global__ void __launch_bounds__(256, 2) su2_measure(const T *__restrict__ U, const T *__restrict__ E, int N,
                                                      double *slots)
{
    const size_t n3 = (size_t)N * N * N;
    const unsigned n3u = (unsigned)n3;  // N <= 1290: below 2^32
    const unsigned un = (unsigned)N, nn = un * un;
    double el = 0.0, mag = 0.0, g2 = 0.0, gmax = 0.0;
    const unsigned stride = gridDim.x * 256u;
    for (unsigned s = blockIdx.x * 256u + threadIdx.x; s < n3u; s += stride) {
        const unsigned row = s / un, x = s - row * un, z = row / un, y = row - z * un;
        const unsigned sp[3] = {x + 1 == un ? s - (un - 1) : s + 1, y + 1 == un ? s - (nn - un) : s + un,
                                z + 1 == un ? s - (n3u - nn) : s + nn};
        const unsigned sm[3] = {x == 0 ? s + (un - 1) : s - 1, y == 0 ? s + (nn - un) : s - un,
                                z == 0 ? s + (n3u - nn) : s - nn};
        Su2Site<T> site;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            site.c[i] = ldU(U, n3, i, s);
            site.m[i] = ldU(U, n3, i, sm[i]);
#pragma unroll
            for (int j = i + 1; j < 3; ++j) {
                site.p[2 * (i + j - 1)] = ldU(U, n3, j, sp[i]);
                site.p[2 * (i + j - 1) + 1] = ldU(U, n3, i, sp[j]);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const T *e = E + (size_t)(3 * i + c) * n3;
                site.e[3 * i + c] = __ldg(e + s);
                site.em[3 * i + c] = __ldg(e + sm[i]);
            }
        }
        const double gg = site.odd() ? site.template add<false>(el, mag) : site.template add<true>(el, mag);
        g2 += gg;
        gmax = fmax(gmax, gg);
    }
    __shared__ double red[8][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v[4] = {el, mag, g2, gmax};
    for (int q = 0; q < 4; ++q) {
        double w = v[q];
        for (int o = 16; o > 0; o >>= 1) {
            const double u = __shfl_xor_sync(0xffffffffu, w, o);
            w = q == 3 ? fmax(w, u) : w + u;
        }
        if (lane == 0) red[warp][q] = w;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double w = red[0][threadIdx.x];
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k)
            w = threadIdx.x == 3 ? fmax(w, red[k][threadIdx.x]) : w + red[k][threadIdx.x];
        slots[4 * blockIdx.x + threadIdx.x] = w;
    }
}

// Sums the slots in a fixed order: warp q of four sums quantity q, lane by lane
// and then across the lanes (one thread adding 608 slots in turn took 146 us).
__global__ void __launch_bounds__(128) su2_sum_slots(const double *slots, int nblocks, double inv_n3, double *out)
{
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double w = 0.0;
    for (int b = lane; b < nblocks; b += 32) w = q == 3 ? fmax(w, slots[4 * b + q]) : w + slots[4 * b + q];
    for (int o = 16; o > 0; o >>= 1) {
        const double u = __shfl_xor_sync(0xffffffffu, w, o);
        w = q == 3 ? fmax(w, u) : w + u;
    }
    if (lane) return;
    if (q == 0) out[0] = 0.5 * w * inv_n3;
    else if (q == 1) out[1] = 2.0 * w * inv_n3;
    else if (q == 2) out[3] = sqrt(w * inv_n3);
    else out[2] = sqrt(w);
}


template <typename T>
__global__ void su2_init(T *U, T *E, int N, uint64_t seed, double amp)
{
    const size_t n3 = (size_t)N * N * N;
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < n3; s += (size_t)gridDim.x * blockDim.x) {
        for (int i = 0; i < 3; ++i) {
            double g[4];
            for (int h = 0; h < 2; ++h) {
                uint64_t w0, w1;
                tl::philox2x64_10(3 * s + i, (1ull << 62) + h, seed, w0, w1);  // random initial links
                const double u1 = ((double)(w0 >> 11) + 1.0) / 9007199254740992.0;
                const double u2 = (double)(w1 >> 11) / 9007199254740992.0;
                const double r = sqrt(-2.0 * log(u1));
                double sn, cs;
                sincospi(2.0 * u2, &sn, &cs);
                g[2 * h] = r * cs;
                g[2 * h + 1] = r * sn;
            }
            const double q1 = amp * g[0], q2 = amp * g[1], q3 = amp * g[2];
            const double inv = 1.0 / sqrt(1.0 + q1 * q1 + q2 * q2 + q3 * q3);
            stU(U, n3, i, s, Q<T>{(T)inv, (T)(q1 * inv), (T)(q2 * inv), (T)(q3 * inv)});
            for (int c = 0; c < 3; ++c) E[(3 * i + c) * n3 + s] = (T)0;
        }
    }
}

// Host layout U[i][c][site] <-> device records U[i][site][c].
template <typename T>
__global__ void su2_to_records(const T *__restrict__ cm, T *__restrict__ rec, size_t n3)
{
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < 3 * n3; k += (size_t)gridDim.x * blockDim.x) {
        const size_t i = k / n3, s = k - i * n3;
        stU(rec, n3, (int)i, s, Q<T>{cm[(4 * i) * n3 + s], cm[(4 * i + 1) * n3 + s], cm[(4 * i + 2) * n3 + s],
                                    cm[(4 * i + 3) * n3 + s]});
    }
}
template <typename T>
__global__ void su2_from_records(const T *__restrict__ rec, T *__restrict__ cm, size_t n3)
{
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < 3 * n3; k += (size_t)gridDim.x * blockDim.x) {
        const size_t i = k / n3, s = k - i * n3;
        const Q<T> q = ldU(rec, n3, (int)i, s);
        cm[(4 * i) * n3 + s] = q.w;
        cm[(4 * i + 1) * n3 + s] = q.x;
        cm[(4 * i + 2) * n3 + s] = q.y;
        cm[(4 * i + 3) * n3 + s] = q.z;
    }
}

}  // namespace

struct tl_su2 {
    int N = 0;
    tl_dtype dtype = TL_F64;
    size_t esz = 8;
    cudaStream_t stream = nullptr;
    void *U[2] = {nullptr, nullptr};
    void *E = nullptr;
    int cur = 0;
    double *slots = nullptr;
    double *out = nullptr;
    int mblocks = 0;
    int sm_count = 0;
    bool has_state = false;
    // the step's tile and launch (su2_plan; grid 0: not planned yet)
    Su2Tile tile{};
    unsigned grid = 0;
    size_t smem = 0;
};

#define SU_CK(call)                                                                                         \
    do {                                                                                                    \
        cudaError_t e_ = (call);                                                                            \
        if (e_ != cudaSuccess)                                                                              \
            return tl::fail(e_ == cudaErrorMemoryAllocation ? TL_ENOMEM : TL_ECUDA, "%s: %s", #call,        \
                            cudaGetErrorString(e_));                                                        \
    } while (0)

namespace {

template <typename T>
using Su2Kernel = void (*)(const T *, T *, T *, int, Su2Tile, T);

bool su2_stages_fields(int N, size_t esz) { return esz == 4 && N % 32 == 0; }

// The code form of a tile: 0 any tile, 1 and 2 the 32 x 8 one without and with
// staged electric fields.  Those measured faster where rows start on a
// 128-byte line (FP32, us: 128^3 76 against 82, 192^3 231 against
// 249, 256^3 532 against 574) and slower elsewhere (100^3 57 against 53, 150^3
// 142 against 130); FP64 has its registers to itself and keeps them there.
template <typename T>
int su2_form(int N, const Su2Tile &t)
{
    return sizeof(T) == 4 && t.tx == 32 && t.ty == 8 ? (su2_stages_fields(N, sizeof(T)) ? 2 : 1) : 0;
}

template <typename T>
Su2Kernel<T> su2_kernel(int form)
{
    if constexpr (sizeof(T) == 4) {
        if (form) return form == 2 ? su2_pass<T, true, true> : su2_pass<T, true, false>;
    }
    return su2_pass<T, false, false>;
}

// Tile shape and grid of the step.  The cost of a tile per plane is its
// warps (and 0.12 of a warp for each warp that forms halo plaquettes), so the
// shape that covers N x N with the fewest warps is taken (of equal ones the
// narrowest): at N = 100, 10 x 25 tiles cover it with 40 CTA-planes of 8 warps where 32 x 8 ones need 52.  FP32
// keeps the 32 x 8 tile with compile-time strides unless the other needs 20%
// fewer warps (100^3: 50 against 53 us; 150^3, 5% fewer: 144 against 130).
//
// Division of the tiles' planes among the CTAs: an even one, every resident
// CTA the same number of planes counted through the tiles, or equal z-chunks
// (waves of CTAs) that keep neighbouring tiles at the same height, so that the
// links they share meet in L2.  FP64 is bound by arithmetic and takes the
// first (100^3 759 against 840 us, 192^3 4950 against 5210); FP32 takes it
// while the links fit in L2 and the estimate is 8% better (128^3 76 against
// 80 us; beyond that size it loses: 192^3 250 against 231, 256^3 572 against 532).
//
// The plan depends on the lattice and the device alone and is kept with the
// lattice.  Every size shares the kernels: their shared-memory limit is raised
// for the largest tile that any lattice has asked for (SmemLimit).
template <typename T>
int su2_plan(tl_su2 *Y)
{
    const int N = Y->N;
    auto shape = [&](int tx, int ty) { return Su2Tile{tx, ty, (N + tx - 1) / tx, (N + ty - 1) / ty, 0}; };
    auto cost = [](const Su2Tile &t) {
        const double warps = (t.tx * t.ty + 31) / 32, halo = (2 * (t.tx + t.ty) + 31) / 32;
        return (double)t.ntx * t.nty * (warps + 0.12 * halo);
    };
    Su2Tile best = shape(32, 8);
    double best_cost = cost(best) * (sizeof(T) == 4 ? 0.8 : 1.0);
    for (int tx = 1; tx <= 64 && tx <= N; ++tx) {
        int ty = 256 / tx;  // the tallest tile of this width, then evened out over N
        while (ty > 1 && ((tx + 2) * (ty + 2) > kSu2MaxHalo || (tx + 1) * (ty + 1) > kSu2MaxPlaq || 2 * (tx + ty) > 256)) --ty;
        const int rows = (N + ty - 1) / ty;
        const Su2Tile t = shape(tx, (N + rows - 1) / rows);
        if ((tx + 2) * (t.ty + 2) <= kSu2MaxHalo && (tx + 1) * (t.ty + 1) <= kSu2MaxPlaq &&
            2 * (tx + t.ty) <= 256 && cost(t) < best_cost)
            best = t, best_cost = cost(t);
    }
    static tl::SmemLimit limit[3];
    const int form = su2_form<T>(N, best);
    const Su2Kernel<T> kern = su2_kernel<T>(form);
    const size_t smem = su2_smem(best.tx, best.ty, sizeof(T), form == 2);
    int per_sm = 0;
    SU_CK(limit[form].raise(kern, smem));
    SU_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem));
    const long slots = (long)(Y->sm_count > 0 ? Y->sm_count : 152) * (per_sm > 0 ? per_sm : 1);
    const long tiles = (long)best.ntx * best.nty, planes = tiles * N;
    // z-chunk: the fewest (waves of CTAs) x (planes per CTA + the ~3 planes of
    // halo copies and the first plane's extra plaquettes)
    long chunk_cost = -1;
    for (int c = N; c >= 1; --c) {
        const long ctas = tiles * ((N + c - 1) / c);
        const long est = (ctas + slots - 1) / slots * (long)(c + 3);
        if (chunk_cost < 0 || est < chunk_cost) chunk_cost = est, best.zc = c;
    }
    unsigned grid = (unsigned)(tiles * ((N + best.zc - 1) / best.zc));
    const long even_cost = (planes + slots - 1) / slots + 4;  // a CTA's range starts one tile and often a second
    const bool in_l2 = 12.0 * N * N * N * sizeof(T) <= 128e6;
    if (sizeof(T) == 8 ? even_cost <= chunk_cost : in_l2 && even_cost < 0.92 * chunk_cost) {
        best.zc = 0;
        grid = (unsigned)(planes < slots ? planes : slots);
    }
    Y->tile = best;
    Y->smem = smem;
    Y->grid = grid;
    return TL_OK;
}

}  // namespace

extern "C" {

void tl_su2_destroy(tl_su2 *Y)
{
    if (!Y) return;
    cudaStreamSynchronize(Y->stream);
    cudaFree(Y->U[0]);
    cudaFree(Y->U[1]);
    cudaFree(Y->E);
    cudaFree(Y->slots);
    cudaFree(Y->out);
    delete Y;
}

int tl_su2_create(tl_su2 **out, int N, tl_dtype dtype, void *cuda_stream)
{
    tl::set_error(TL_OK, "", "");
    if (!out) return tl::fail(TL_EINVAL, "NULL out");
    *out = nullptr;
    if (N < 4 || N > 1290) return tl::fail(TL_EINVAL, "N must be in [4, 1290]");
    if (dtype != TL_F32 && dtype != TL_F64) return tl::fail(TL_EINVAL, "unknown dtype");
    tl_su2 *Y = new (std::nothrow) tl_su2();
    if (!Y) return tl::fail(TL_ENOMEM, "host allocation failed");
    Y->N = N;
    Y->dtype = dtype;
    Y->esz = dtype == TL_F32 ? 4 : 8;
    Y->stream = static_cast<cudaStream_t>(cuda_stream);
    const size_t n3 = (size_t)N * N * N;
    const size_t need = 33 * n3 * Y->esz;  // two link buffers (12 values a site each) and the fields (9)
    size_t free_b = 0;
    if (tl::free_device_bytes(need + (64u << 20), &free_b) != cudaSuccess) {
        delete Y;
        return tl::fail(TL_ECUDA, "cudaMemGetInfo failed (no CUDA device?)");
    }
    if (need + (64u << 20) > free_b) {
        delete Y;
        return tl::fail(TL_ENOMEM, "SU(2) lattice needs %zu bytes", need);
    }
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&Y->sm_count, cudaDevAttrMultiProcessorCount, dev);
    Y->mblocks = 4 * (Y->sm_count > 0 ? Y->sm_count : 152);
    cudaError_t e = tl::device_alloc(&Y->U[0], 12 * n3 * Y->esz);
    if (e == cudaSuccess) e = tl::device_alloc(&Y->U[1], 12 * n3 * Y->esz);
    if (e == cudaSuccess) e = tl::device_alloc(&Y->E, 9 * n3 * Y->esz);
    if (e == cudaSuccess) e = tl::device_alloc(&Y->slots, sizeof(double) * 4 * Y->mblocks);
    if (e == cudaSuccess) e = tl::device_alloc(&Y->out, sizeof(double) * 4);
    if (e != cudaSuccess) {
        tl_su2_destroy(Y);
        return tl::fail(TL_ENOMEM, "SU(2) allocation: %s", cudaGetErrorString(e));
    }
    *out = Y;
    return TL_OK;
}

int tl_su2_set_state(tl_su2 *Y, const void *U, const void *E)
{
    tl::set_error(TL_OK, "", "");
    if (!Y || !U || !E) return tl::fail(TL_EINVAL, "NULL argument");
    const size_t n3 = (size_t)Y->N * Y->N * Y->N;
    // host links into the spare buffer, then transposed into records
    SU_CK(cudaMemcpyAsync(Y->U[Y->cur ^ 1], U, 12 * n3 * Y->esz, cudaMemcpyHostToDevice, Y->stream));
    if (Y->dtype == TL_F32)
        su2_to_records<float><<<Y->mblocks, 256, 0, Y->stream>>>(static_cast<const float *>(Y->U[Y->cur ^ 1]),
                                                                 static_cast<float *>(Y->U[Y->cur]), n3);
    else
        su2_to_records<double><<<Y->mblocks, 256, 0, Y->stream>>>(static_cast<const double *>(Y->U[Y->cur ^ 1]),
                                                                  static_cast<double *>(Y->U[Y->cur]), n3);
    SU_CK(cudaGetLastError());
    SU_CK(cudaMemcpyAsync(Y->E, E, 9 * n3 * Y->esz, cudaMemcpyHostToDevice, Y->stream));
    SU_CK(cudaStreamSynchronize(Y->stream));
    Y->has_state = true;
    return TL_OK;
}

int tl_su2_get_state(tl_su2 *Y, void *U, void *E)
{
    tl::set_error(TL_OK, "", "");
    if (!Y || (!U && !E)) return tl::fail(TL_EINVAL, "NULL argument");
    const size_t n3 = (size_t)Y->N * Y->N * Y->N;
    if (U) {  // records transposed into the spare buffer, then copied out
        if (Y->dtype == TL_F32)
            su2_from_records<float><<<Y->mblocks, 256, 0, Y->stream>>>(static_cast<const float *>(Y->U[Y->cur]),
                                                                       static_cast<float *>(Y->U[Y->cur ^ 1]), n3);
        else
            su2_from_records<double><<<Y->mblocks, 256, 0, Y->stream>>>(static_cast<const double *>(Y->U[Y->cur]),
                                                                        static_cast<double *>(Y->U[Y->cur ^ 1]), n3);
        SU_CK(cudaGetLastError());
        SU_CK(cudaMemcpyAsync(U, Y->U[Y->cur ^ 1], 12 * n3 * Y->esz, cudaMemcpyDeviceToHost, Y->stream));
    }
    if (E) SU_CK(cudaMemcpyAsync(E, Y->E, 9 * n3 * Y->esz, cudaMemcpyDeviceToHost, Y->stream));
    SU_CK(cudaStreamSynchronize(Y->stream));
    return TL_OK;
}

int tl_su2_init_random(tl_su2 *Y, uint64_t seed, double amp)
{
    tl::set_error(TL_OK, "", "");
    if (!Y || !(amp >= 0.0)) return tl::fail(TL_EINVAL, "bad argument");
    if (Y->dtype == TL_F32)
        su2_init<float><<<Y->mblocks, 256, 0, Y->stream>>>(static_cast<float *>(Y->U[Y->cur]),
                                                           static_cast<float *>(Y->E), Y->N, seed, amp);
    else
        su2_init<double><<<Y->mblocks, 256, 0, Y->stream>>>(static_cast<double *>(Y->U[Y->cur]),
                                                            static_cast<double *>(Y->E), Y->N, seed, amp);
    SU_CK(cudaGetLastError());
    Y->has_state = true;
    return TL_OK;
}

int tl_su2_step(tl_su2 *Y, int n, double dt)
{
    tl::NvtxScope nvtx_range("tl_su2_step");
    tl::set_error(TL_OK, "", "");
    if (!Y) return tl::fail(TL_EINVAL, "NULL lattice");
    if (n < 0 || !isfinite(dt) || dt == 0.0) return tl::fail(TL_EINVAL, "n >= 0 and a finite nonzero dt needed");
    if (!Y->has_state) return tl::fail(TL_ESTATE, "no state");
    if (!Y->grid) {
        const int rc = Y->dtype == TL_F32 ? su2_plan<float>(Y) : su2_plan<double>(Y);
        if (rc) return rc;
    }
    auto steps = [&](auto value) -> int {
        using S = decltype(value);
        const Su2Kernel<S> kern = su2_kernel<S>(su2_form<S>(Y->N, Y->tile));
        for (int k = 0; k < n; ++k) {
            kern<<<Y->grid, 256, Y->smem, Y->stream>>>(static_cast<const S *>(Y->U[Y->cur]),
                                                       static_cast<S *>(Y->U[Y->cur ^ 1]), static_cast<S *>(Y->E), Y->N,
                                                       Y->tile, (S)dt);
            SU_CK(cudaGetLastError());
            Y->cur ^= 1;
        }
        return TL_OK;
    };
    return Y->dtype == TL_F32 ? steps(0.0f) : steps(0.0);
}

int tl_su2_measure(tl_su2 *Y, double *out4)
{
    tl::NvtxScope nvtx_range("tl_su2_measure");
    tl::set_error(TL_OK, "", "");
    if (!Y || !out4) return tl::fail(TL_EINVAL, "NULL argument");
    const size_t n3 = (size_t)Y->N * Y->N * Y->N;
    const int mgrid = Y->mblocks / 2;  // two CTAs per SM, all resident
    if (Y->dtype == TL_F32)
        su2_measure<float><<<mgrid, 256, 0, Y->stream>>>(static_cast<const float *>(Y->U[Y->cur]),
                                                              static_cast<const float *>(Y->E), Y->N, Y->slots);
    else
        su2_measure<double><<<mgrid, 256, 0, Y->stream>>>(static_cast<const double *>(Y->U[Y->cur]),
                                                               static_cast<const double *>(Y->E), Y->N, Y->slots);
    SU_CK(cudaGetLastError());
    su2_sum_slots<<<1, 128, 0, Y->stream>>>(Y->slots, mgrid, 1.0 / (double)n3, Y->out);
    SU_CK(cudaGetLastError());
    SU_CK(cudaMemcpyAsync(out4, Y->out, 4 * sizeof(double), cudaMemcpyDeviceToHost, Y->stream));
    SU_CK(cudaStreamSynchronize(Y->stream));
    return TL_OK;
}

}  // extern "C"
