// Device scratch of tl_init_fluctuations and tl_spectrum: stream-ordered
// allocations from one memory pool per device, private to the library.
//
// The device's default pool gives its memory back at every synchronisation, so
// that each tl_spectrum mapped its scratch anew: 0.7-0.8 ms per call at 256^3,
// a quarter of the call.  This pool keeps up to kKeepBytes between calls
// (256^3 needs 135 MB, 384^3 453 MB; larger scratch is returned as before).
// What it keeps is given back when the device's last lattice is destroyed, and
// whenever the library itself runs short of device memory (scratch_release).
// Allocation and free are ordered on the caller's stream, and the driver orders
// reuse across streams, so threads and streams share the pool safely.
#include <mutex>

#include "tl_internal.cuh"

namespace {

constexpr int kMaxDevices = 64;
constexpr cuuint64_t kKeepBytes = 1ull << 30;

std::mutex g_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};
int g_users[kMaxDevices] = {};

}  // namespace

namespace tl {

cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t s)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    cudaMemPool_t pool;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_pool[dev]) {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t made;
            if ((e = cudaMemPoolCreate(&made, &props)) != cudaSuccess) return e;
            cuuint64_t keep = kKeepBytes;
            if ((e = cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
                cudaMemPoolDestroy(made);
                return e;
            }
            g_pool[dev] = made;
        }
        pool = g_pool[dev];
    }
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    scratch_release(dev);  // what the pool keeps may be in other pieces
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

cudaError_t device_alloc_bytes(void **p, size_t bytes)
{
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return e;
    scratch_release(dev);
    return cudaMalloc(p, bytes);
}

void scratch_release(int dev)
{
    if (dev < 0 || dev >= kMaxDevices) return;
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_pool[dev]) cudaMemPoolTrimTo(g_pool[dev], 0);
}

void scratch_user(int dev, int change)
{
    if (dev < 0 || dev >= kMaxDevices) return;
    std::lock_guard<std::mutex> lk(g_mu);
    g_users[dev] += change;
    if (g_users[dev] == 0 && g_pool[dev]) cudaMemPoolTrimTo(g_pool[dev], 0);
}

cudaError_t free_device_bytes(size_t need, size_t *free_b)
{
    size_t total = 0;
    cudaError_t e = cudaMemGetInfo(free_b, &total);
    if (e != cudaSuccess || need <= *free_b) return e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    scratch_release(dev);
    return cudaMemGetInfo(free_b, &total);
}

}  // namespace tl
