#include "device_memory.h"

#include <mutex>

#include "kernels.h"

namespace spmm {

namespace {

cudaError_t device_pool(cudaMemPool_t* pool) {
    static std::mutex mu;
    static cudaMemPool_t pools[kMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        e = cudaMemPoolCreate(&p, &props);
        if (e != cudaSuccess) return e;
        unsigned long long keep = kPoolKeepBytes;
        e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return e;
        }
        pools[dev] = p;
    }
    *pool = pools[dev];
    return cudaSuccess;
}

}  // namespace

cudaError_t dev_alloc(void** ptr, size_t bytes, cudaStream_t stream) {
    *ptr = nullptr;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = device_pool(&pool);
    if (e != cudaSuccess) return e;
    if (bytes == 0) bytes = 16;
    e = cudaMallocFromPoolAsync(ptr, bytes, pool, stream);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(ptr, bytes, pool, stream);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *ptr = nullptr;
    }
    return e;
}

cudaError_t dev_alloc_ready(void** ptr, size_t bytes, cudaStream_t stream) {
    cudaError_t e = dev_alloc(ptr, bytes, stream);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        dev_free(*ptr, stream);
        *ptr = nullptr;
    }
    return e;
}

void dev_free(void* ptr, cudaStream_t stream) {
    if (ptr) cudaFreeAsync(ptr, stream);
}

void dev_give_back(size_t keep) {
    cudaMemPool_t pool = nullptr;
    unsigned long long reserved = 0;
    if (device_pool(&pool) != cudaSuccess ||
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess || reserved <= keep)
        return;
    cudaStreamSynchronize(nullptr);              // the frees count once they are known to have happened
    cudaMemPoolTrimTo(pool, keep);
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
