"""The integer conversions between FP32 and FP64 (csrc/tl_bits.cuh) compiled for
the host: the same bits as the language's conversions, over every exponent,
ties, carries, subnormals, zeros, infinities; a NaN stays one."""
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
#define __device__
#define __forceinline__ inline
template <typename A, typename B> static A as(B b) { A a; static_assert(sizeof a == sizeof b, ""); memcpy(&a, &b, sizeof a); return a; }
static unsigned __float_as_uint(float v) { return as<unsigned>(v); }
static float __uint_as_float(unsigned v) { return as<float>(v); }
static int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static int __double2hiint(double v) { return (int)(as<uint64_t>(v) >> 32); }
static int __double2loint(double v) { return (int)(uint32_t)as<uint64_t>(v); }
static double __hiloint2double(int hi, int lo) { return as<double>((uint64_t)(uint32_t)hi << 32 | (uint32_t)lo); }
#include "tl_bits.cuh"
static long bad;
static void widen(uint32_t b)
{
    const float v = as<float>(b);
    const double got = tl::widen_bits(v);
    bad += isnan(v) ? !isnan(got) : as<uint64_t>(got) != as<uint64_t>((double)v);
}
static void narrow(uint64_t b)
{
    const double v = as<double>(b);
    const float got = tl::narrow_bits(v);
    bad += isnan(v) ? !isnan(got) : as<uint32_t>(got) != as<uint32_t>((float)v);
    bad += as<uint64_t>(tl::flip(v, true)) != (b ^ 1ull << 63) || as<uint64_t>(tl::flip(v, false)) != b;
}
int main()
{
    uint64_t x = 88172645463325252ull;
    for (unsigned e = 0; e < 512; ++e)
        for (unsigned i = 0; i < 512; ++i) {
            x ^= x << 13, x ^= x >> 7, x ^= x << 17;
            const unsigned m = i < 24 ? 1u << i : i < 48 ? (1u << (i - 24)) - 1 : (unsigned)x;
            widen(e << 23 | (m & 0x7fffffu));
        }
    for (uint64_t e = 0; e < 4096; ++e)
        for (unsigned i = 0; i < 512; ++i) {
            x ^= x << 13, x ^= x >> 7, x ^= x << 17;
            const uint64_t m = i < 53 ? 1ull << i : i < 106 ? (1ull << (i - 53)) - 1 : i < 159 ? ~0ull << (i - 106)
                               : i < 220 ? (x & ~0x1fffffffull) | 1ull << 28 : i < 250 ? (x & ~0x1fffffffull) + (1ull << 28) - 1 : x;
            narrow(e << 52 | (m & 0xfffffffffffffull));
        }
    printf("%ld\n", bad);
    return 0;
}
"""


def test_integer_conversions_equal_the_languages(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2607_24908_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    assert int(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout) == 0
