#include "fr_pool.h"

#include <mutex>

namespace {

constexpr int MAXDEV = 64;
std::mutex g_mutex;
cudaMemPool_t g_pool[MAXDEV] = {};

// the current device's pool, made on first use (`make`); null if there is none
cudaMemPool_t pool_of_device(bool make) {
    int dev = 0, ok = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAXDEV) return nullptr;
    std::lock_guard<std::mutex> lock(g_mutex);
    if (g_pool[dev] || !make) return g_pool[dev];
    if (cudaDeviceGetAttribute(&ok, cudaDevAttrMemoryPoolsSupported, dev) != cudaSuccess || !ok) return nullptr;
    cudaMemPoolProps pr = {};
    pr.allocType = cudaMemAllocationTypePinned;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &pr) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    unsigned long long keep = POOL_KEEP;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        cudaMemPoolDestroy(pool);
        return nullptr;
    }
    return g_pool[dev] = pool;
}

}  // namespace

bool fr_pool_alloc(void** p, size_t n, cudaStream_t s) {
    *p = nullptr;
    cudaMemPool_t pool = pool_of_device(true);
    if (!pool) return false;
    if (cudaMallocFromPoolAsync(p, n, pool, s) == cudaSuccess) return true;
    cudaGetLastError();
    *p = nullptr;
    return false;
}

void fr_pool_free(void* p, cudaStream_t s) {
    if (p) cudaFreeAsync(p, s);
}

void fr_pool_trim() {
    cudaMemPool_t pool = pool_of_device(false);
    if (pool && cudaMemPoolTrimTo(pool, 0) != cudaSuccess) cudaGetLastError();
}
