#include "fr_pool.h"

#include <cuda.h>

#include <map>
#include <mutex>

namespace {

std::mutex g_mutex;
std::map<unsigned long long, cudaMemPool_t> g_pool;   // by context

// The current context's id: unique for the life of the process, so that it differs
// after cudaDeviceReset, which ends a device's context and the pools made in it
// (their handles are then never used again).  0: unknown.
unsigned long long context_id() {
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    static const GetId get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? reinterpret_cast<GetId>(f) : nullptr;
    }();
    unsigned long long id = 0;
    if (!get) return 0;
    if (get(nullptr, &id) == CUDA_SUCCESS) return id;
    // this thread has no context yet, or one that was reset: the runtime makes one
    if (cudaFree(nullptr) != cudaSuccess || get(nullptr, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// the current context's pool, made on first use (`make`); null if there is none
cudaMemPool_t pool_of_context(bool make) {
    const unsigned long long ctx = context_id();
    int dev = 0, ok = 0;
    if (ctx == 0 || cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lock(g_mutex);
    const auto at = g_pool.find(ctx);
    if (at != g_pool.end() || !make) return at != g_pool.end() ? at->second : nullptr;
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
    return g_pool[ctx] = pool;
}

}  // namespace

bool fr_pool_alloc(void** p, size_t n, cudaStream_t s) {
    *p = nullptr;
    cudaMemPool_t pool = pool_of_context(true);
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
    cudaMemPool_t pool = pool_of_context(false);
    if (pool && cudaMemPoolTrimTo(pool, 0) != cudaSuccess) cudaGetLastError();
}
