"""The table form of Box-Muller's logarithm and circle (csrc/tl_boxmuller.cuh)
compiled for the host and compared with long double over random uniforms, the
table's edges, the smallest uniforms and those next to one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
struct double2 { double x, y; };
#define __device__
#define __forceinline__ inline
#define __syncthreads()
static double __longlong_as_double(long long v) { double d; memcpy(&d, &v, 8); return d; }
static int __clzll(long long v) { return __builtin_clzll(v); }
static struct { int x; } threadIdx{0}, blockDim{1};
#include "tl_boxmuller.cuh"
static tl::BoxMullerTable t;
static double log_worst, circle_worst;
static int negative;
static void check_log(uint64_t m)
{
    const long double ref = -logl((long double)m / 9007199254740992.0L);
    const double got = tl::neg_log_u53(&t, m);
    negative += !(got >= 0.0);
    const double e = ref == 0 ? (got != 0.0) : (double)fabsl((got - ref) / ref);
    if (!(e <= log_worst)) log_worst = e;
}
static void check_circle(uint64_t m)
{
    const long double a = 2.0L * acosl(-1.0L) * ((long double)m / 9007199254740992.0L);
    double c, s;
    tl::unit_circle_u53(&t, m, c, s);
    const double e = (double)fmaxl(fabsl(c - cosl(a)), fabsl(s - sinl(a)));
    if (!(e <= circle_worst)) circle_worst = e;
}
int main()
{
    tl::load_box_muller(&t);
    const uint64_t one = 1ull << 53;
    for (uint64_t i = 0; i < 4096; ++i) check_log(1 + i), check_log(one - i);
    for (int bit = 0; bit < 53; ++bit)
        for (uint64_t j = 0; j <= 128; ++j)
            for (int d = -1; d <= 1; ++d) {
                const uint64_t m = (1ull << bit) + (bit >= 7 ? j << (bit - 7) : 0) + d;
                if (m >= 1 && m <= one) check_log(m);
            }
    for (uint64_t j = 0; j <= 512; ++j)
        for (int d = -2; d <= 2; ++d) check_circle(((j << 44) + d) & (one - 1));
    uint64_t x = 88172645463325252ull;
    for (int i = 0; i < 2000000; ++i) {
        x ^= x << 13, x ^= x >> 7, x ^= x << 17;
        check_log((x >> 11) + 1), check_circle(x >> 11);
    }
    printf("%.17g %.17g %d\n", log_worst, circle_worst, negative);
    return 0;
}
"""


def test_table_box_muller_is_accurate_to_a_few_ulp(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "bm"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-O2", "-std=gnu++17", "-I", os.path.join(ROOT, "paper_2607_24908_gb300", "csrc"),
                           str(src), "-o", str(exe)])
    log_worst, circle_worst, negative = (float(v) for v in subprocess.check_output([str(exe)]).split())
    # the logarithm: half an ulp each (2^-53) from r, the polynomial, the table point and two
    # sums, the first of them up to twice the result; the circle: table point, two products, sum
    assert log_worst <= 6 * 2.0 ** -53 and negative == 0
    assert circle_worst <= 3 * 2.0 ** -53
