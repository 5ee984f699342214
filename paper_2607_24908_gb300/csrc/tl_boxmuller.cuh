// The two FP64 functions of Box-Muller, -ln u and (cos, sin) 2 pi u of 53-bit
// uniforms, by table and short polynomial.
//
// The Gaussian draws (initial modes, FP64 Langevin noise) are bound by GB300's
// FP64 pipe, two operations a clock per SM.  A library logarithm and sincospi
// reduce their arguments in FP64 and evaluate long polynomials, about 80
// operations together; a uniform is an integer over 2^53, so the reductions
// here are integer instructions (another pipe), a table entry takes the
// argument near zero, and 11 and 14 operations remain.  The logarithm is
// Tang's scheme (P. T. P. Tang, "Table-driven implementation of the logarithm
// function in IEEE floating-point arithmetic", ACM TOMS 16, 1990): u = 2^k z,
// ln u = k ln 2 + ln c + log1p(z/c - 1) with c a table point near z.
//
// Accuracy against extended precision over 2 10^7 uniforms, half of them next to one:
// -ln u to 3.2e-16 of itself (rms 6.8e-17; a library logarithm 1.1e-16 and
// 4.6e-17), the circle to 2.4e-16 (rms 5.4e-17; cos(2 pi u) of a rounded product:
// 6.4e-16, rms 1.6e-16), and the Gaussian they make, sqrt(-2 ln u) cos(2 pi v), to
// 4.1e-16 of its modulus (rms 7.5e-17) where the library's forms gave 7.0e-16 (rms
// 1.7e-16).
#pragma once

#include <math.h>
#include <stdint.h>

namespace tl {

constexpr int kLogEntries = 128, kCircleEntries = 256;
constexpr int kLogUpper = 43;  // table index from which z is halved

struct BoxMullerTable {
    double2 log[kLogEntries];        // (1/c, ln c)
    double2 circle[kCircleEntries];  // (cos, sin) of 2 pi j/256
};

namespace detail {

// ln v for v in (1/2, 2) with v - 1 exact: 2 atanh((v - 1)/(v + 1)), rounded once
// but for 2^-5 of an ulp: the quotient's own error is added to the series' tail.
constexpr double low_half(double v)  // what a 26-bit upper half leaves (T. J. Dekker, Numer. Math. 18, 1971)
{
    const double c = 134217729.0 * v;  // 2^27 + 1
    return v - (c - (c - v));
}
constexpr double log_near_one(double v)
{
    const double n = v - 1.0, d = v + 1.0, dl = v - (d - 1.0);  // v + 1 = d + dl
    const double s = n / d, s2 = s * s;
    const double sl = low_half(s), sh = s - sl, el = low_half(d), eh = d - el;
    const double rest = ((n - sh * eh) - sh * el - sl * eh) - sl * el - s * dl;  // n - s (d + dl)
    double sum = 0.0;
    for (int i = 41; i >= 3; i -= 2) sum = sum * s2 + 1.0 / i;
    return 2.0 * s + 2.0 * (s * s2 * sum + rest / d * (1.0 + s2));
}
// cos and sin of 2 pi j/256, |j| <= 32, by their series.
constexpr double cos_turn(int j)
{
    const double x = 2.0 * M_PI * j / 256.0, x2 = x * x;
    double sum = 1.0;
    for (int i = 20; i >= 2; i -= 2) sum = 1.0 - sum * x2 / (i * (i - 1.0));
    return sum;
}
constexpr double sin_turn(int j)
{
    const double x = 2.0 * M_PI * j / 256.0, x2 = x * x;
    double sum = 1.0;
    for (int i = 21; i >= 3; i -= 2) sum = 1.0 - sum * x2 / (i * (i - 1.0));
    return x * sum;
}

// alignas: load_box_muller reads it in 16-byte words.
struct alignas(16) RawTable {
    double log[kLogEntries][2] = {};
    double circle[kCircleEntries][2] = {};
    constexpr RawTable()
    {
        // z in [1, 1.336) as it is and above halved, so that u near 1 is z
        // near 1 with k = 0; there c = 1 keeps the logarithm's relative accuracy
        // (the place of the cut: k ln 2 and ln c cancel least)
        for (int j = 0; j < kLogEntries; ++j) {
            const double mid = (1.0 + (j + 0.5) / kLogEntries) * (j < kLogUpper ? 1.0 : 0.5);
            const bool one = j == 0 || j == kLogEntries - 1;
            log[j][0] = one ? 1.0 : 1.0 / mid;
            log[j][1] = one ? 0.0 : -log_near_one(log[j][0]);
        }
        for (int j = 0; j < kCircleEntries; ++j) {
            const int quarter = (j + 32) / 64 % 4, d = j - (j + 32) / 64 * 64;  // |d| <= 32
            const double c = cos_turn(d), s = sin_turn(d);
            circle[j][0] = quarter == 0 ? c : quarter == 1 ? -s : quarter == 2 ? -c : s;
            circle[j][1] = quarter == 0 ? s : quarter == 1 ? c : quarter == 2 ? -s : -c;
        }
    }
};

}  // namespace detail

static_assert(alignof(detail::RawTable) >= alignof(double2) && sizeof(detail::RawTable) == sizeof(BoxMullerTable),
              "the raw table is copied as double2");
static __device__ const detail::RawTable g_box_muller{};

// Copies the table into a CTA's shared memory (ends with a barrier).
__device__ __forceinline__ void load_box_muller(BoxMullerTable *t)
{
    const double2 *src = reinterpret_cast<const double2 *>(&g_box_muller);
    double2 *dst = reinterpret_cast<double2 *>(t);
    for (int i = threadIdx.x; i < kLogEntries + kCircleEntries; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
}

// (double)k for |k| < 64, by integer instructions (a conversion holds the FP64 pipe).
__device__ __forceinline__ double small_int(int k)
{
    const int a = k < 0 ? -k : k;
    const int lead = 63 - __clzll((long long)a | 1);  // of 0: 0, with the bit removed below
    const uint64_t bits = ((uint64_t)(1023 + lead) << 52) + (((uint64_t)(a - (1 << lead))) << (52 - lead));
    return __longlong_as_double((long long)((a ? bits : 0) | (k < 0 ? 1ull << 63 : 0)));
}

// -ln(m 2^-53) for an integer 1 <= m <= 2^53.
__device__ __forceinline__ double neg_log_u53(const BoxMullerTable *t, uint64_t m)
{
    const int lead = __clzll((long long)m);
    const uint64_t frac = (m << lead) << 1;  // the bits below the leading one
    const int j = (int)(frac >> 57), upper = j >= kLogUpper;
    const double z = __longlong_as_double((long long)((uint64_t)(0x3ff - upper) << 52 | frac >> 12));
    const int k = 10 - lead + upper;  // u = 2^k z
    const double2 e = t->log[j];
    const double r = fma(z, e.x, -1.0);
    double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    q = fma(r, q, 1.0 / 5.0);
    q = fma(r, q, -1.0 / 4.0);
    q = fma(r, q, 1.0 / 3.0);
    q = fma(r, q, -1.0 / 2.0);
    // the small terms first: one rounding at the size of the result
    return fma(small_int(-k), M_LN2, -(e.y + fma(r * r, q, r)));
}

// (cos, sin)(2 pi m 2^-53) for an integer 0 <= m < 2^53.
__device__ __forceinline__ void unit_circle_u53(const BoxMullerTable *t, uint64_t m, double &c, double &s)
{
    const uint64_t a = m + (1ull << 44);  // to the nearest of 256 points
    const double2 e = t->circle[(a >> 45) & 255];
    // the rest as 2^52 + (rest + 2^44), exactly, less the two
    const double d = __longlong_as_double((long long)(0x4330000000000000ull | (a & ((1ull << 45) - 1)))) -
                     (4503599627370496.0 + 17592186044416.0);
    const double x = d * (2.0 * M_PI / 9007199254740992.0), x2 = x * x;  // |x| < 0.0123
    const double sd = fma(x * x2, fma(x2, fma(x2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), x);
    const double cd = x2 * fma(x2, fma(x2, -1.0 / 720.0, 1.0 / 24.0), -0.5);  // cos - 1
    c = fma(-e.y, sd, fma(e.x, cd, e.x));
    s = fma(e.x, sd, fma(e.y, cd, e.y));
}

}  // namespace tl
