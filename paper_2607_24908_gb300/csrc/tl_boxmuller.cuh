// The two FP64 functions of Box-Muller, -ln u and (cos, sin) 2 pi u of 53-bit
// uniforms, by table and short polynomial.
//
// The Gaussian draws (initial modes, FP64 Langevin noise) are bound by GB300's
// FP64 pipe, two operations a clock per SM.  A library logarithm and sincospi
// reduce their arguments in FP64 and evaluate long polynomials, about 80
// operations together; a uniform is an integer over 2^53, so the reductions
// here are integer instructions (another pipe), a table entry takes the
// argument near zero, and 13 and 16 operations remain.  The logarithm is
// Tang's scheme (P. T. P. Tang, "Table-driven implementation of the logarithm
// function in IEEE floating-point arithmetic", ACM TOMS 16, 1990): u = 2^k z,
// ln u = k ln 2 + ln c + log1p(z/c - 1) with c a table point near z.
//
// The table's values carry their own roundings' rest, and what is of the size of the
// result is rounded once.  Accuracy against extended precision over 2 10^7 uniforms, half
// of them next to one: -ln u to 2.3e-16 of itself (rms 4.8e-17; a library logarithm
// 1.1e-16 and 4.6e-17), the circle to 5.7e-17, and the Gaussian they make, sqrt(-2 ln u)
// cos(2 pi v), to 3.1e-16 of its modulus (rms 5.6e-17, that of correctly rounded
// functions; with sincos of a rounded 2 pi v 7.0e-16, rms 1.7e-16).
#pragma once

#include <math.h>
#include <stdint.h>

namespace tl {

constexpr int kLogEntries = 128, kCircleEntries = 256;
constexpr int kLogUpper = 43;  // table index from which z is halved

struct BoxMullerTable {
    double2 log[kLogEntries];        // (1/c, ln c to a multiple of 2^-43)
    double2 circle[kCircleEntries];  // (cos, sin) of 2 pi j/256
    double2 circle_low[kCircleEntries];  // what their rounding left
    double log_low[kLogEntries];         // the rest of ln c
};

namespace detail {

// The table's values, in pairs hi + lo of about 2^-104 (T. J. Dekker, "A floating-point
// technique for extending the available precision", Numer. Math. 18, 1971).
struct Sum {
    double hi, lo;
};
constexpr Sum sum_of(double a, double b)
{
    const double s = a + b, t = s - a;
    return Sum{s, (a - (s - t)) + (b - t)};
}
constexpr Sum add(Sum a, Sum b)
{
    const Sum s = sum_of(a.hi, b.hi);
    return sum_of(s.hi, s.lo + (a.lo + b.lo));
}
constexpr Sum product(double a, double b)
{
    const double c = 134217729.0 * a, d = 134217729.0 * b, p = a * b;  // 2^27 + 1
    const double ah = c - (c - a), al = a - ah, bh = d - (d - b), bl = b - bh;
    return Sum{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr Sum mul(Sum a, Sum b)
{
    const Sum p = product(a.hi, b.hi);
    return sum_of(p.hi, p.lo + (a.hi * b.lo + a.lo * b.hi));
}
constexpr Sum div(Sum a, Sum b)
{
    const double q = a.hi / b.hi;
    const Sum p = mul(Sum{q, 0.0}, b);
    return sum_of(q, ((a.hi - p.hi) + (a.lo - p.lo)) / b.hi);
}
constexpr Sum of(double v) { return Sum{v, 0.0}; }
constexpr Sum upper_bits(Sum v)  // hi a multiple of 2^-43
{
    const double hi = (double)(long long)(v.hi * 0x1p43) * 0x1p-43;
    return Sum{hi, (v.hi - hi) + v.lo};
}
// ln v for v in (1/2, 2): 2 atanh((v - 1)/(v + 1)).
constexpr Sum log_near_one(double v)
{
    const Sum s = div(sum_of(v, -1.0), sum_of(v, 1.0)), s2 = mul(s, s);
    Sum sum{};
    for (int i = 41; i >= 1; i -= 2) sum = add(mul(sum, s2), div(of(1.0), of(i)));
    return upper_bits(mul(mul(of(2.0), s), sum));
}
// ln 2 (M_LN2 and what it lacks); cosine and sine of 2 pi j/256, |j| <= 32, by their series.
constexpr Sum kLn2 = upper_bits(Sum{M_LN2, 2.3190468138462996e-17});
constexpr Sum turn(int j) { return mul(Sum{M_PI, 1.2246467991473532e-16}, of(j / 128.0)); }
constexpr Sum cos_turn(int j)
{
    const Sum x = turn(j), x2 = mul(x, x);
    Sum sum = of(1.0);
    for (int i = 22; i >= 2; i -= 2) sum = add(of(1.0), mul(mul(sum, x2), div(of(-1.0), of(i * (i - 1.0)))));
    return sum;
}
constexpr Sum sin_turn(int j)
{
    const Sum x = turn(j), x2 = mul(x, x);
    Sum sum = of(1.0);
    for (int i = 23; i >= 3; i -= 2) sum = add(of(1.0), mul(mul(sum, x2), div(of(-1.0), of(i * (i - 1.0)))));
    return mul(x, sum);
}

// alignas: load_box_muller reads it in 16-byte words.
struct alignas(16) RawTable {
    double log[kLogEntries][2] = {};
    double circle[kCircleEntries][2] = {};
    double circle_low[kCircleEntries][2] = {};
    double log_low[kLogEntries] = {};
    constexpr RawTable()
    {
        // z in [1, 1.336) as it is and above halved, so that u near 1 is z
        // near 1 with k = 0; there c = 1 keeps the logarithm's relative accuracy
        // (the place of the cut: k ln 2 and ln c cancel least)
        for (int j = 0; j < kLogEntries; ++j) {
            const double mid = (1.0 + (j + 0.5) / kLogEntries) * (j < kLogUpper ? 1.0 : 0.5);
            const bool one = j == 0 || j == kLogEntries - 1;
            log[j][0] = one ? 1.0 : 1.0 / mid;
            const Sum ln = log_near_one(log[j][0]);  // of 1/c
            log[j][1] = one ? 0.0 : -ln.hi;
            log_low[j] = one ? 0.0 : -ln.lo;
        }
        for (int j = 0; j < kCircleEntries; ++j) {
            const int quarter = (j + 32) / 64 % 4, d = j - (j + 32) / 64 * 64;  // |d| <= 32
            const Sum c = cos_turn(d), s = sin_turn(d), &x = quarter % 2 ? s : c, &y = quarter % 2 ? c : s;
            const double sx = quarter == 1 || quarter == 2 ? -1.0 : 1.0, sy = quarter >= 2 ? -1.0 : 1.0;
            circle[j][0] = sx * x.hi, circle_low[j][0] = sx * x.lo;
            circle[j][1] = sy * y.hi, circle_low[j][1] = sy * y.lo;
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
    for (int i = threadIdx.x; i < (int)(sizeof(BoxMullerTable) / sizeof(double2)); i += blockDim.x) dst[i] = src[i];
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
    // the upper parts add up exactly, so that one rounding is of the size of the result
    const double nk = small_int(-k);
    return fma(nk, detail::kLn2.hi, -e.y) + (fma(nk, detail::kLn2.lo, -t->log_low[j]) - fma(r * r, q, r));
}

// (cos, sin)(2 pi m 2^-53) for an integer 0 <= m < 2^53.
__device__ __forceinline__ void unit_circle_u53(const BoxMullerTable *t, uint64_t m, double &c, double &s)
{
    const uint64_t a = m + (1ull << 44);  // to the nearest of 256 points
    const int j = (int)(a >> 45) & 255;
    const double2 e = t->circle[j], low = t->circle_low[j];
    // the rest as 2^52 + (rest + 2^44), exactly, less the two
    const double d = __longlong_as_double((long long)(0x4330000000000000ull | (a & ((1ull << 45) - 1)))) -
                     (4503599627370496.0 + 17592186044416.0);
    const double x = d * (2.0 * M_PI / 9007199254740992.0), x2 = x * x;  // |x| < 0.0123
    const double sd = fma(x * x2, fma(x2, fma(x2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), x);
    const double cd = x2 * fma(x2, fma(x2, -1.0 / 720.0, 1.0 / 24.0), -0.5);  // cos - 1
    c = e.x + fma(-e.y, sd, fma(e.x, cd, low.x));
    s = e.y + fma(e.x, sd, fma(e.y, cd, low.y));
}

}  // namespace tl
