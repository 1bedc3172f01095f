// Device memory of the library: every allocation and release goes through here.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

namespace spmv {

// With the environment variable SPMV_FAULT_ALLOC=k, the k-th allocation of an
// entry-point call returns cudaErrorMemoryAllocation without allocating (the
// call must then return SPMV_ERR_OOM and release what it had allocated).
cudaError_t dev_malloc(void **p, size_t bytes);
cudaError_t dev_malloc_async(void **p, size_t bytes, cudaStream_t s);
template <typename T>
inline cudaError_t dev_malloc(T **p, size_t bytes) {
    return dev_malloc(reinterpret_cast<void **>(p), bytes);
}
template <typename T>
inline cudaError_t dev_malloc_async(T **p, size_t bytes, cudaStream_t s) {
    return dev_malloc_async(reinterpret_cast<void **>(p), bytes, s);
}
// starts the count of a call's allocations
void reset_alloc_count();

// Frees what dev_malloc gave (null is fine).  The block may still be in use by
// work already launched: it is handed out again only after the device has been
// waited for.
void dev_free(void *p);
// Waits for the device's work; blocks freed before are then handed out again.
void dev_settle();
// Gives back what is kept of the current context, after the device's work is done.
cudaError_t dev_trim();

}  // namespace spmv
