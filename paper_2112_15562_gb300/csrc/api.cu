// Error reporting and library metadata.
#include <stdio.h>

#include <map>
#include <mutex>
#include <string>

#include "gj_internal.h"

namespace gj {

static thread_local std::string g_last_error;

void set_error(const std::string &msg) { g_last_error = msg; }

gj_status cuda_fail(cudaError_t e, const char *what) {
    std::string m = std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
    set_error(m);
    cudaGetLastError();  // reported here: the next call's launches do not find it again
    return e == cudaErrorMemoryAllocation ? GJ_ERR_OOM : GJ_ERR_CUDA;
}

std::mutex &capture_mutex() {
    static std::mutex mu;
    return mu;
}
cudaError_t sync_device() {
    std::lock_guard<std::mutex> lock(capture_mutex());
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

constexpr uint64_t kPoolKeep = 128 << 20;  // (a pool reserves memory in pieces of 32 MB)
static cudaMemPool_t own_pool(int dev) {
    static std::mutex mu;
    static std::map<int, cudaMemPool_t> pools;
    std::lock_guard<std::mutex> lock(mu);
    auto it = pools.find(dev);
    if (it != pools.end()) return it->second;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = kPoolKeep;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();
        pool = nullptr;
    } else if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        cudaMemPoolDestroy(pool);
        pool = nullptr;
    }
    pools[dev] = pool;
    return pool;
}
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t st) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (cudaMemPool_t pool = own_pool(dev)) return cudaMallocFromPoolAsync(p, bytes, pool, st);
    return cudaMallocAsync(p, bytes, st);
}

}  // namespace gj

extern "C" const char *gj_last_error(void) { return gj::g_last_error.c_str(); }

extern "C" const char *gj_version(void) { return "gj 0.1 (sm_103a)"; }
