"""The form of the library's Philox-2x64-10 for first counter words below 2^32
(csrc/tl_philox.cuh) equals the general form, compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <stdio.h>
#include "tl_philox.cuh"
int main()
{
    const uint32_t edge[] = {0u, 1u, 2u, 0x7fffffffu, 0x80000000u, 0xfffffffeu, 0xffffffffu};
    uint64_t x = 88172645463325252ull;
    int n = 0;
    for (int i = 0; i < 20000; ++i) {
        x ^= x << 13, x ^= x >> 7, x ^= x << 17;
        const uint32_t c0 = i < 7 ? edge[i] : (uint32_t)x;
        const uint64_t c1 = x * 0x9E3779B97F4A7C15ull, key = ~x;
        uint64_t a, b, c, d;
        tl::philox2x64_10((uint64_t)c0, c1, key, a, b);
        tl::philox2x64_10_low(c0, c1, key, c, d);
        n += a != c || b != d;
    }
    printf("%d\n", n);
    return 0;
}
"""


def test_low_counter_form_is_the_general_one(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "low"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2607_24908_gb300", "csrc"),
                           str(src), "-o", str(exe)])
    assert subprocess.check_output([str(exe)]).split() == [b"0"]
