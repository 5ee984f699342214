"""A kernel's dynamic shared-memory limit is shared by all lattices and threads: it
is only ever raised (csrc/tl_smem.cuh).  Compiled for the host against a fake of
the runtime that makes one thread's smaller request come after another's larger
one has been set, wherever it can."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_24908_gb300", "csrc")

FAKE = r"""
#pragma once
#include <atomic>
#include <chrono>
#include <thread>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidDevice = 101 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
inline std::atomic<int> limit{0}, large_set{0}, calls{0};
inline cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
template <typename K>
cudaError_t cudaFuncSetAttribute(K, cudaFuncAttribute, int bytes)
{
    ++calls;
    if (bytes < 100)  // a small request: let a large one of another thread through first, if it can come
        for (int i = 0; i < 300 && !large_set; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(1));
    limit = bytes;
    if (bytes >= 100) large_set = 1;
    return cudaSuccess;
}
"""

MAIN = r"""
#include <stdio.h>
#include "tl_smem.cuh"
static void kernel() {}
static tl::SmemLimit lim;
int main()
{
    std::thread small([] { lim.raise(kernel, 90); });
    std::this_thread::sleep_for(std::chrono::milliseconds(50));
    std::thread large([] { lim.raise(kernel, 120); });
    small.join();
    large.join();
    const int both = limit, n = calls;
    lim.raise(kernel, 60), lim.raise(kernel, 120), lim.raise(kernel, 0);
    printf("%d %d %d\n", both, (int)limit, (int)calls - n);
    return 0;
}
"""


def test_the_limit_is_never_lowered(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    src, exe = tmp_path / "main.cpp", tmp_path / "limit"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-std=gnu++17", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(src), "-o", str(exe)])
    both, after, further = (int(v) for v in subprocess.check_output([str(exe)]).split())
    assert both == 120 and after == 120 and further == 0


def test_every_kernels_limit_goes_through_it():
    for name in glob.glob(os.path.join(CSRC, "*.cu*")):
        if os.path.basename(name) == "tl_smem.cuh":
            continue
        with open(name) as f:
            assert "cudaFuncSetAttribute" not in re.sub(r"//[^\n]*", "", f.read()), name
