// The library's device-memory pools.  Host code only.
#include "pool.cuh"

#include <mutex>

namespace lsq {

// The pools, by device.  A pool that no longer works (the device was reset) is made again; what
// the dead one held went with the device's context.
namespace {
std::mutex g_pool_mu;
cudaMemPool_t g_pool[64] = {};
// The device's pool, made if there is none.  `failed` is a pool that refused an allocation: it is
// replaced if it is still the device's and does not answer any more.  A live pool refuses for the
// caller's reason (a stream that is not one, say) and stays: *out is `failed` again.
cudaError_t pool_of(int dev, cudaMemPool_t failed, cudaMemPool_t* out) {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (failed && g_pool[dev] == failed) {
        uint64_t keep = 0;
        if (cudaMemPoolGetAttribute(failed, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaGetLastError();
            g_pool[dev] = nullptr;
        }
    }
    if (!g_pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t made = nullptr;
        cudaError_t e = cudaMemPoolCreate(&made, &props);
        if (e != cudaSuccess) return e;
        uint64_t keep = POOL_KEEP;
        e = cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(made);
            return e;
        }
        g_pool[dev] = made;
    }
    *out = g_pool[dev];
    return cudaSuccess;
}
}  // namespace

cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t st) {
    *p = nullptr;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaMemPool_t pool = nullptr;
    if (dev >= 64 || pool_of(dev, nullptr, &pool) != cudaSuccess) {
        cudaGetLastError();
        return cudaMallocAsync(p, bytes, st);   // no pool of our own: the device's
    }
    e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    } else if (e == cudaErrorInvalidValue || e == cudaErrorInvalidResourceHandle) {
        cudaGetLastError();
        cudaMemPool_t now = nullptr;
        cudaError_t made = pool_of(dev, pool, &now);
        if (made != cudaSuccess) return made;
        if (now != pool) e = cudaMallocFromPoolAsync(p, bytes, now, st);
    }
    return e;
}

void pool_free(int device, std::initializer_list<void*> ptrs) {
    bool any = false;
    for (void* p : ptrs) any = any || p != nullptr;
    if (!any) return;
    int current = -1;
    if (cudaGetDevice(&current) != cudaSuccess) return;
    if (current != device && cudaSetDevice(device) != cudaSuccess) return;
    cudaDeviceSynchronize();
    for (void* p : ptrs)
        if (p) cudaFreeAsync(p, 0);
    if (current != device) cudaSetDevice(current);
}

}  // namespace lsq
