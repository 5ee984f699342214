// A kernel's limit of dynamic shared memory (host side).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <atomic>
#include <mutex>

namespace tl {

// The limit is an attribute of the kernel on a device, shared by every lattice
// and thread that launches it, so it is only ever raised: whatever a thread has
// asked for stays allowed until its launch.  One object per kernel.  Compared and
// set under a mutex; a request within what is set takes one atomic load.
class SmemLimit {
    static constexpr int kDevices = 64;
    std::atomic<size_t> set_[kDevices] = {};
    std::mutex mu_;

public:
    template <typename K>
    cudaError_t raise(K kern, size_t smem)
    {
        if (smem == 0) return cudaSuccess;
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kDevices) return cudaErrorInvalidDevice;
        std::atomic<size_t> &set = set_[dev];
        if (smem <= set.load(std::memory_order_acquire)) return cudaSuccess;
        std::lock_guard<std::mutex> lk(mu_);
        if (smem <= set.load(std::memory_order_relaxed)) return cudaSuccess;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) set.store(smem, std::memory_order_release);
        return e;
    }
};

}  // namespace tl
