"""The table of Box-Muller (csrc/tl_boxmuller.cuh) is copied in 16-byte words: with
double2 aligned as on the device, the static table starts on a 16-byte boundary."""
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
struct alignas(16) double2 { double x, y; };
#define __device__
#define __forceinline__ inline
#define __syncthreads()
static double __longlong_as_double(long long v) { double d; memcpy(&d, &v, 8); return d; }
static int __clzll(long long v) { return __builtin_clzll(v); }
static struct { int x; } threadIdx{0}, blockDim{1};
#include "tl_boxmuller.cuh"
int main()
{
    printf("%zu %zu\n", alignof(tl::detail::RawTable), alignof(tl::BoxMullerTable));
    return 0;
}
"""


def test_raw_table_is_aligned_to_its_16_byte_reads(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "layout"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-std=gnu++17", "-I", os.path.join(ROOT, "paper_2607_24908_gb300", "csrc"), str(src),
                           "-o", str(exe)])
    raw, table = (int(v) for v in subprocess.check_output([str(exe)]).split())
    assert raw >= table == 16
