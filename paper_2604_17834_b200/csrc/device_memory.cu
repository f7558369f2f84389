#include "device_memory.h"

#include <mutex>

#include "kernels.h"

namespace spmm {

namespace {

struct Pool {
    cudaMemPool_t pool = nullptr;
    cudaStream_t service = nullptr;      // carries allocations only (dev_alloc_ready): never waits for a user's work
};

cudaError_t device_pool(Pool* pool) {
    static std::mutex mu;
    static Pool pools[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!pools[dev].pool) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        Pool p;
        e = cudaMemPoolCreate(&p.pool, &props);
        if (e != cudaSuccess) return e;
        unsigned long long keep = kPoolKeepBytes;
        e = cudaMemPoolSetAttribute(p.pool, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p.service, cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(p.pool);
            return e;
        }
        pools[dev] = p;
    }
    *pool = pools[dev];
    return cudaSuccess;
}

// `stream` null with `ready`: the service stream, waited for.
cudaError_t alloc_from_pool(void** ptr, size_t bytes, cudaStream_t stream, bool ready) {
    *ptr = nullptr;
    Pool pool;
    cudaError_t e = device_pool(&pool);
    if (e != cudaSuccess) return e;
    if (ready) stream = pool.service;
    if (bytes == 0) bytes = 16;
    e = cudaMallocFromPoolAsync(ptr, bytes, pool.pool, stream);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        cudaMemPoolTrimTo(pool.pool, 0);
        e = cudaMallocFromPoolAsync(ptr, bytes, pool.pool, stream);
    }
    if (e == cudaSuccess && ready) {
        e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) cudaFreeAsync(*ptr, stream);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *ptr = nullptr;
    }
    return e;
}

}  // namespace

cudaError_t dev_alloc(void** ptr, size_t bytes, cudaStream_t stream) { return alloc_from_pool(ptr, bytes, stream, false); }

cudaError_t dev_alloc_ready(void** ptr, size_t bytes) { return alloc_from_pool(ptr, bytes, nullptr, true); }

void dev_free(void* ptr, cudaStream_t stream) {
    if (ptr) cudaFreeAsync(ptr, stream);
}

void dev_give_back(size_t keep) {
    Pool pool;
    unsigned long long reserved = 0;
    if (device_pool(&pool) != cudaSuccess ||
        cudaMemPoolGetAttribute(pool.pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess || reserved <= keep)
        return;
    cudaStreamSynchronize(nullptr);              // the frees count once they are known to have happened
    cudaMemPoolTrimTo(pool.pool, keep);
}

cudaError_t dev_malloc(void** ptr, size_t bytes) {
    if (bytes == 0) bytes = 16;
    cudaError_t e = cudaMalloc(ptr, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        dev_give_back(0);
        e = cudaMalloc(ptr, bytes);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *ptr = nullptr;
    }
    return e;
}

}  // namespace spmm
