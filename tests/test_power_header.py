"""Whole powers of the scale factor (csrc/tl_power.cuh) compiled for the host: each
within the roundings of its own multiplications and of one reciprocal, over the
exponents that whole alpha in -4 .. 6 gives, far outside FP32's range included."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#define __device__
#define __forceinline__ inline
#include "tl_power.cuh"
static double worst[32];
static void check(double x)
{
    for (int n = -11; n <= 13; ++n) {
        long double p = 1.0L;
        for (int i = 0; i < (n < 0 ? -n : n); ++i) p *= (long double)x;
        const long double ref = n < 0 ? 1.0L / p : p;
        if (!(fabsl(ref) > 1e-300L && fabsl(ref) < 1e300L)) continue;
        const double e = (double)fabsl(((long double)tl::int_power(x, n) - ref) / ref);
        if (!(e <= worst[n + 11])) worst[n + 11] = e;
    }
}
int main()
{
    uint64_t s = 88172645463325252ull;
    for (int i = 0; i < 400000; ++i) {
        s ^= s << 13, s ^= s >> 7, s ^= s << 17;
        const double u = (double)(s >> 11) / 9007199254740992.0;
        check(0.99 + 0.02 * u), check(exp(9.0 * u)), check(1.0 / (1.0 + 9.0 * u)), check(exp(120.0 * (u - 0.5)));
    }
    for (int n = -11; n <= 13; ++n) printf("%d %.17g\n", n, worst[n + 11]);
    return 0;
}
"""


def test_powers_carry_only_their_own_roundings(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "power"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-O2", "-std=gnu++17", "-I", os.path.join(ROOT, "paper_2607_24908_gb300", "csrc"),
                           str(src), "-o", str(exe)])
    u = 2.0 ** -53
    for line in subprocess.check_output([str(exe)], text=True).splitlines():
        n, e = line.split()
        # |n| - 1 roundings of a product tree (a square counts its operand's twice), one of
        # the reciprocal; 1% for the second order and the iteration's own error
        roundings = max(abs(int(n)) - 1, 0) + (1 if int(n) < 0 else 0)
        assert float(e) <= 1.01 * roundings * u, (n, float(e) / u)
