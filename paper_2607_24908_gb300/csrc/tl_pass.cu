// Launch geometry, variant dispatch and the background-reset kernel of the
// fused pass (the kernels themselves are in tl_pass_impl.cuh, instantiated
// per precision in tl_pass_f32.cu and tl_pass_f64.cu).
#include <math.h>

#include "tl_internal.cuh"
#include "tl_scale.cuh"

namespace tl {

__global__ void set_background_kernel(Model m, Scalars *sc, double a, double b)  // one warp
{
    if (m.expanding) write_scale_powers(m, sc, a, a, a);
    if (threadIdx.x != 0) return;
    if (m.expanding) {
        sc->a = a;
        sc->b = b;
    } else {
        sc->a = 1.0;
        sc->b = 0.0;
        for (int i = 0; i < kScalePowers; ++i) (&sc->wl)[i] = 1.0;
    }
    sc->drift = 0.0;
    sc->pending_dt = 0.0;
    sc->time = 0.0;
    sc->hubble = 0.0;
    sc->status = TL_OK;
    sc->ticket = 0u;
    for (int i = 0; i < kMaxQ; ++i) sc->E[i] = 0.0;
}

// ---- tile rows and z-chunks of the streaming kernel ----------------------------
//
// FP64 passes are bound by the FP64 pipe, where a warp's instruction holds its SM
// for 16 clocks whatever its lanes do, so that a pass takes as long as the SM
// with the most warp-planes: per warp and plane about 50 instructions a field (57
// in chunks of one plane, which drift three planes for one), and per CTA its
// sums and latencies, about 60.  That estimate gives the rows of thin tiles: 32^3 takes
// tiles of 16 x 8 threads on 128 SMs, not 16 x 16 on 64.

constexpr int kThinChunk = 3;  // chunks up to here may have tiles of fewer rows

static double f64_cost(int N, int gx, int txt, int ty, int zc, int sms)
{
    const long ctas = (long)gx * ((N + ty - 1) / ty) * ((N + zc - 1) / zc);
    int warps = (txt * ty + 31) / 32;
    if (warps < 4) warps = 4;  // fewer do not fill the pipe: an operation's result takes 65 clocks
    return (double)((ctas + sms - 1) / sms) * (warps * ((zc == 1 ? 57 : 50 * zc) + 10) + 60);
}

// Rows of an FP64 tile of zc planes: all that fit, or in thin chunks, which are
// for lattices that do not fill the GPU, the cheapest number.
static int f64_tile_rows(int N, int gx, int txt, int ty_max, int zc, int sms)
{
    int best = ty_max;
    if (zc <= kThinChunk)
        for (int ty = ty_max - 1; ty >= 1; --ty)
            if (f64_cost(N, gx, txt, ty, zc, sms) < f64_cost(N, gx, txt, best, zc, sms)) best = ty;
    return best;
}

// FP64 chunk (shared_tile): the cheapest by (waves of two
// CTAs per SM) x (warps per CTA x planes), where a last wave of at most one CTA per
// SM counts 0.6 and a CTA no less than 6 warps.  Over 36 lattices of 32^3 to 384^3 the
// choice is 0.6% slower than the best of a sweep (8% at 144^3 with two fields), that
// of the estimate above 5% (us: 144^3 155 -> 127, 160^3 199 -> 160, 212^3 396 -> 355, 300^3
// 1090 -> 932; three fields 160^3 636 -> 501).  Two fields keep 32 planes from 128^3
// to 508^3 unless another is estimated 4% cheaper: estimates that close do not tell
// (the estimate's choice / 32 planes: 288^3 1859 / 1903, 312^3 2226 / 2194, 368^3 3621 /
// 3615, 448^3 6215 / 6336, 508^3 9187 / 9153).  From 512^3 on they do (512^3 9182 / 9247,
// 536^3 11403 / 11439, 576^3 13089 / 13173, 640^3 17983 / 18117).
static double f64_shared_cost(int N, int gx, int txt, int ty, int zc, int sms)
{
    const long ctas = (long)gx * ((N + ty - 1) / ty) * ((N + zc - 1) / zc), last = ctas % (2 * sms);
    const double waves = (double)(ctas / (2 * sms)) + (last == 0 ? 0.0 : last <= sms ? 0.6 : 1.0);
    int warps = (txt * ty + 31) / 32;
    if (warps < 6) warps = 6;
    return waves * (warps * (zc + 0.3) + 3.0);
}

static int f64_chunk(int N, int nf, int gx, int txt, int ty_max, int sms)
{
    auto cost = [&](int zc) {
        return f64_shared_cost(N, gx, txt, f64_tile_rows(N, gx, txt, ty_max, zc, sms), zc, sms);
    };
    int best = N >= 128 ? 32 : 1;
    double least = cost(best) * (N >= 128 && N < 512 && nf == 2 ? 0.96 : 1.0);
    for (int zc = 1; zc <= N && zc <= 128; ++zc)
        if (cost(zc) < least) least = cost(zc), best = zc;
    return best;
}

// FP32 chunk.  Below 192^3 the pass runs out of L2 and its time is latency and
// the last CTA's sum over all others: the shortest chunk whose CTAs are all on
// the GPU at once, one per SM while that is at most six field-planes, else two
// per SM (us, two fields: 48^3 11.0 -> 9.7 with 1 plane, not 3, 64^3 12.0 -> 10.0 with
// 2, not 4, 128^3 25.7 -> 20.3 with 7, not 4, 160^3 61 -> 44 with 16, not 4).
// Larger lattices: at least four planes (the planes on either side of a chunk are
// traffic) and several waves of CTAs.
static int f32_chunk(int N, int nf, int tiles, int sms)
{
    if (N < 192) {
        auto shortest = [&](long ctas) {
            int zc = 1;
            while (zc < N && (long)tiles * ((N + zc - 1) / zc) > ctas) ++zc;
            return zc;
        };
        const int zc = shortest(sms);
        return zc * nf <= 6 ? zc : shortest(2L * sms);
    }
    int zc = 128;
    while (zc > 4 && (long)tiles * ((N + zc - 1) / zc) < 8L * sms) zc /= 2;
    return zc;
}

PassGeom pass_geometry(int N, int elem_bytes, int sm_count, int nf, const PassTuning &t)
{
    const int W = 16 / elem_bytes;
    PassGeom g;
    const int per_row = N / W;  // N % 4 == 0 is required, so W | N
    g.variant = t.variant;
    g.cwarps = (t.variant == kVariantTma) ? (t.cwarps == 15 ? 15 : 7) : 8;
    // CTAs of whole warps (the CTA reduction needs them) whose compute threads
    // are laid over a tile of txt x ty threads; leftover threads idle.
    g.threads = (t.variant == kVariantLdg && t.threads == 512) ? 512 : 256;
    const int threads = t.variant == kVariantTma ? 32 * g.cwarps : g.threads;
    const int txt_max = (t.variant == kVariantLdg && (t.txt == 8 || t.txt == 16)) ? t.txt : 32;
    g.tile_x = g.txt = per_row < txt_max ? per_row : txt_max;
    if (txt_max == 32 && (t.variant == kVariantLdg || N < kFullRowTiles)) g.txt = even_row_tile(per_row);
    g.ty = threads / g.txt;
    if (g.ty > N) g.ty = N;
    const int gx = (per_row + g.txt - 1) / g.txt;
    int gy = (N + g.ty - 1) / g.ty;
    const int sms = sm_count > 0 ? sm_count : 152;
    const bool f64_stream = t.variant == kVariantLdg && elem_bytes == 8;
    int zc = t.zc;
    if (zc <= 0) {
        if (f64_stream) {
            zc = f64_chunk(N, nf, gx, g.txt, g.ty, sms);
        } else if (t.variant == kVariantLdg) {
            zc = f32_chunk(N, nf, gx * gy, sms);
        } else {  // TMA: long enough to amortise the two extra planes, short enough for several waves
            zc = N < 128 ? N : 128;
            while (zc > 4 && (long)gx * gy * ((N + zc - 1) / zc) < 8L * sms) zc /= 2;
        }
    }
    if (zc > N) zc = N;
    g.zc = zc;
    if (f64_stream) {
        g.ty = f64_tile_rows(N, gx, g.txt, g.ty, zc, sms);
        gy = (N + g.ty - 1) / g.ty;
    }
    g.grid = dim3(gx, gy, (N + zc - 1) / zc);
    g.nblocks = g.grid.x * g.grid.y * g.grid.z;
    g.stages = 0;
    g.smem = 0;
    g.prefetch = 0;
    if (g.variant == kVariantLdg) {
        g.prefetch = (t.prefetch > 0 && g.threads == 256) ? 3 : 0;
        g.smem = (size_t)g.prefetch * nf * 2 * 256 * 16;
    }
    g.lpad = 128 / elem_bytes;
    if (g.variant == kVariantTma) {
        // ring depth: as deep as fits two CTAs per SM (<= 113 KB each), at
        // least 3 (two planes read + one in flight), at most 8; each stage
        // holds 2 nf slots of tma_slot_bytes.
        const size_t per_stage = (size_t)nf * 2 * tma_slot_bytes(g.txt, g.ty);
        int S = t.stages > 0 ? t.stages : 8;
        if (S > 8) S = 8;
        // two CTAs per SM for 7 compute warps, one for 15
        const size_t cap = (t.stages > 0 || g.cwarps > 7 ? 227u : 113u) * 1024u;
        while (S > 3 && per_stage * S > cap) --S;
        g.stages = S;
        g.smem = per_stage * S;
    }
    return g;
}

cudaError_t launch_pass_f32(const Model &m, const FieldPtrs &fp, const PassCoef &c, const PassGeom &g, Scalars *sc,
                            double *slots, bool measure_only, cudaStream_t s, const TmaMaps *maps);
cudaError_t launch_pass_f64(const Model &m, const FieldPtrs &fp, const PassCoef &c, const PassGeom &g, Scalars *sc,
                            double *slots, bool measure_only, cudaStream_t s, const TmaMaps *maps);

cudaError_t launch_pass(int dtype, const Model &m, const FieldPtrs &fp, const PassCoef &c, const PassGeom &g,
                        Scalars *sc, double *slots, bool measure_only, cudaStream_t s, const TmaMaps *maps)
{
    if (m.nf < 1 || m.nf > kMaxFields) return cudaErrorInvalidValue;
    return dtype == TL_F32 ? launch_pass_f32(m, fp, c, g, sc, slots, measure_only, s, maps)
                           : launch_pass_f64(m, fp, c, g, sc, slots, measure_only, s, maps);
}

cudaError_t launch_group_f32(int nf, int variant, int prefetch, int stages, size_t smem, const BatchJob *jobs,
                             const unsigned *first_item, int njobs, unsigned total, const PassCoef &c, int grid,
                             cudaStream_t s);
cudaError_t launch_group_f64(int nf, int variant, int prefetch, int stages, size_t smem, const BatchJob *jobs,
                             const unsigned *first_item, int njobs, unsigned total, const PassCoef &c, int grid,
                             cudaStream_t s);

cudaError_t launch_group(int dtype, int nf, int variant, int prefetch, int stages, size_t smem, const BatchJob *jobs,
                         const unsigned *first_item, int njobs, unsigned total, const PassCoef &c, int grid,
                         cudaStream_t s)
{
    return dtype == TL_F32
               ? launch_group_f32(nf, variant, prefetch, stages, smem, jobs, first_item, njobs, total, c, grid, s)
               : launch_group_f64(nf, variant, prefetch, stages, smem, jobs, first_item, njobs, total, c, grid, s);
}

size_t tma_group_smem(int nf, int stages, int max_txt, int max_ty)
{
    return (size_t)stages * nf * 2 * tma_slot_bytes(max_txt, max_ty);
}

// Refresh the ghost rows of one array (layout in tl_internal.cuh): the rows
// above and below every plane, copies of rows N - 1 and 0.
template <typename T>
__global__ void fill_ghosts_y(T *a, int N, long long P, long long PP)
{
    const long long n = (long long)N * N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        T *plane = a + (i / N) * PP;
        const long long x = i % N;
        plane[-P + x] = plane[(long long)(N - 1) * P + x];
        plane[(long long)N * P + x] = plane[x];
    }
}

cudaError_t launch_fill_ghosts(int dtype, void *origin, int N, long long P, long long PP, cudaStream_t s)
{
    const long long n = (long long)N * N;
    const unsigned grid = (unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
    if (dtype == TL_F32)
        fill_ghosts_y<float><<<grid, 256, 0, s>>>(static_cast<float *>(origin), N, P, PP);
    else
        fill_ghosts_y<double><<<grid, 256, 0, s>>>(static_cast<double *>(origin), N, P, PP);
    return cudaGetLastError();
}

cudaError_t launch_set_background(const Model &m, Scalars *sc, double a, double b, cudaStream_t s)
{
    set_background_kernel<<<1, 32, 0, s>>>(m, sc, a, b);
    return cudaGetLastError();
}

}  // namespace tl
