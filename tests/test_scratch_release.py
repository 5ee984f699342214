"""What the scratch pool keeps between calls is given back when the library runs short
of device memory (csrc/tl_scratch.cu), compiled for the host against a fake of the
runtime: a device of 100 units of which the pool holds some unused."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_24908_gb300", "csrc")

FAKE = r"""
#pragma once
#include <stddef.h>
#include <stdint.h>
enum cudaError_t { cudaSuccess = 0, cudaErrorMemoryAllocation = 2, cudaErrorInvalidDevice = 101 };
enum { cudaMemAllocationTypePinned = 1, cudaMemLocationTypeDevice = 1, cudaMemPoolAttrReleaseThreshold = 4 };
typedef uint64_t cuuint64_t;
typedef void *cudaStream_t;
typedef struct Pool *cudaMemPool_t;
struct cudaMemPoolProps { int allocType; struct { int type, id; } location; };
extern size_t used, pool_unused;
extern int errors_pending;
const size_t kDevice = 100;
inline cudaError_t fake_short() { ++errors_pending; return cudaErrorMemoryAllocation; }
inline cudaError_t cudaGetLastError() { errors_pending = 0; return cudaSuccess; }
inline cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
inline cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t)&used; return cudaSuccess; }
inline cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, int, void *) { return cudaSuccess; }
inline cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
inline cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep) { if (pool_unused > keep) pool_unused = keep; return cudaSuccess; }
inline cudaError_t cudaMalloc(void **p, size_t n)
{
    if (used + pool_unused + n > kDevice) return fake_short();
    used += n;
    *p = &used;
    return cudaSuccess;
}
// the unused memory of the pool is in pieces too small for any request
inline cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return cudaMalloc(p, n); }
inline cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = kDevice - used - pool_unused; *t = kDevice; return cudaSuccess; }
namespace tl {
cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t s);
void scratch_release(int dev);
void scratch_user(int dev, int change);
cudaError_t free_device_bytes(size_t need, size_t *free_b);
cudaError_t device_alloc_bytes(void **p, size_t bytes);
}
"""

MAIN = r"""
#include <stdio.h>
#include "tl_internal.cuh"
size_t used, pool_unused;
int errors_pending;
int main()
{
    void *p = nullptr;
    tl::scratch_user(0, 1);
    int ok = tl::scratch_alloc(&p, 10, nullptr) == cudaSuccess;  // makes the pool
    pool_unused = 50;
    ok = ok && tl::device_alloc_bytes(&p, 60) == cudaSuccess && pool_unused == 0;
    pool_unused = 20;
    ok = ok && tl::scratch_alloc(&p, 25, nullptr) == cudaSuccess && pool_unused == 0;
    ok = ok && errors_pending == 0;
    // truly short: refused, as without the pool
    pool_unused = 5;
    ok = ok && tl::device_alloc_bytes(&p, 6) == cudaErrorMemoryAllocation;
    ok = ok && tl::scratch_alloc(&p, 6, nullptr) == cudaErrorMemoryAllocation;
    pool_unused = 5;
    tl::scratch_user(0, -1);
    printf("%d\n", ok && pool_unused == 0);
    return 0;
}
"""


def test_memory_the_pool_keeps_is_given_back_when_it_is_short(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "tl_internal.cuh").write_text(FAKE)
    shutil.copy(os.path.join(CSRC, "tl_scratch.cu"), tmp_path / "tl_scratch.cpp")
    (tmp_path / "main.cpp").write_text(MAIN)
    subprocess.check_call([cxx, "-std=gnu++17", str(tmp_path / "main.cpp"), str(tmp_path / "tl_scratch.cpp"), "-o",
                           str(tmp_path / "scratch")])
    assert subprocess.check_output([str(tmp_path / "scratch")]).split() == [b"1"]
