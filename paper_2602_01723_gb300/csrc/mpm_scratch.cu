// mpm_scratch.cu -- the memory pool behind mpm_scratch.h
#include "mpm_scratch.h"

#include <mutex>

namespace mpm {

namespace {

constexpr int MAX_DEVICES = 64;
std::mutex g_mutex;
cudaMemPool_t g_pool[MAX_DEVICES] = {};

// the pool of a device, made on first use; NULL when it cannot be made
cudaMemPool_t pool_of(int device) {
    std::lock_guard<std::mutex> lock(g_mutex);
    if (device < 0 || device >= MAX_DEVICES) return nullptr;
    if (!g_pool[device]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        cudaMemPool_t p = nullptr;
        unsigned long long keep = SCRATCH_KEEP;
        if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaGetLastError();
            cudaMemPoolDestroy(p);
            return nullptr;
        }
        g_pool[device] = p;
    }
    return g_pool[device];
}

}  // namespace

cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t st) {
    int device = -1;
    if (cudaGetDevice(&device) == cudaSuccess) {
        const cudaMemPool_t pool = pool_of(device);
        if (pool) {
            const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
            if (e == cudaSuccess) return e;
            // out of memory: what this pool keeps in pieces too small goes back, and
            // the default pool may hold memory that another user has freed into it
            if (e == cudaErrorMemoryAllocation) cudaMemPoolTrimTo(pool, 0);
        }
    }
    cudaGetLastError();
    return cudaMallocAsync(p, bytes, st);
}

void scratch_trim() {
    std::lock_guard<std::mutex> lock(g_mutex);
    for (cudaMemPool_t p : g_pool)
        if (p && cudaMemPoolTrimTo(p, 0) != cudaSuccess) cudaGetLastError();
}

cudaError_t device_alloc(void **p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        scratch_trim();
        e = cudaMalloc(p, bytes);
    }
    return e;
}

}  // namespace mpm
