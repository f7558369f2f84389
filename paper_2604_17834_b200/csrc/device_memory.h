// Device memory of the library: stream-ordered allocations from one pool per device.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

namespace spmm {

// Building a handle takes some thirty device arrays and destroying it gives them back; with cudaMalloc and
// cudaFree (a synchronisation each) they were most of the 8.9 ms that building, running and destroying a
// WCSR handle of 780 K nonzeros took (destroying alone 0.91 ms, 0.03 with the pool).  Between handles the pool
// keeps at most this many bytes per device: what it holds beyond them goes back to the device when a handle is
// destroyed (dev_give_back), and all that is free when an allocation of the library fails.  CUDA orders reuse:
// memory freed on one stream is handed to another only once the work before the free has completed.
constexpr size_t kPoolKeepBytes = size_t{256} << 20;

// Like cudaMalloc for use on `stream` (after it has been synchronised: anywhere); bytes = 0 gives a valid
// small allocation.  The current device's pool.
cudaError_t dev_alloc(void** ptr, size_t bytes, cudaStream_t stream);
// The same, and `stream` is synchronised: ready for every stream when the call returns (as after cudaMalloc), for
// memory that a handle keeps, whose runs may come on any stream.  (A stream of the library's own in its place need
// not wait for the caller's work, but does not reuse what was freed on the others.)
cudaError_t dev_alloc_ready(void** ptr, size_t bytes, cudaStream_t stream);
// Null is accepted.  The memory must not be in use by work outside `stream`'s order.
void dev_free(void* ptr, cudaStream_t stream);
// After frees on the default stream: what the pool holds beyond kPoolKeepBytes and nobody uses goes back to the
// device before this returns, so that others can allocate it.  keep: 0 gives back all that is free.
void dev_give_back(size_t keep = kPoolKeepBytes);
// cudaMalloc for memory outside the pool; what the pool has free is given back before it fails.
cudaError_t dev_malloc(void** ptr, size_t bytes);

template <class T>
inline bool dev_alloc_ok(T** ptr, size_t bytes, cudaStream_t stream) {
    return dev_alloc(reinterpret_cast<void**>(ptr), bytes, stream) == cudaSuccess;
}

template <class T>
inline bool dev_alloc_ready_ok(T** ptr, size_t bytes, cudaStream_t stream) {
    return dev_alloc_ready(reinterpret_cast<void**>(ptr), bytes, stream) == cudaSuccess;
}

}  // namespace spmm
