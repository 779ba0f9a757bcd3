// Every allocation of the library.  The CUDA runtime keeps the error of a
// refused allocation until it is read, and a launch helper that ends with
// cudaGetLastError() would report it for its own, successful launch: a caller
// that goes on after a refusal (an executor serving a block's requests in groups, a
// fusion that does without a buffer) would fail for no reason.  So a refusal is
// returned and not left behind; *p is null after it.
#pragma once

#include <cstddef>

#include <cuda_runtime_api.h>

namespace pvs {

inline cudaError_t taken(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

template <typename T>
cudaError_t device_alloc(T** p, size_t count) {
    void* v = nullptr;
    const cudaError_t e = taken(cudaMalloc(&v, (count ? count : 1) * sizeof(T)));
    *p = e == cudaSuccess ? static_cast<T*>(v) : nullptr;
    return e;
}

// Pinned host memory.
template <typename T>
cudaError_t pinned_alloc(T** p, size_t count) {
    void* v = nullptr;
    const cudaError_t e = taken(cudaMallocHost(&v, (count ? count : 1) * sizeof(T)));
    *p = e == cudaSuccess ? static_cast<T*>(v) : nullptr;
    return e;
}

// Stream-ordered, from `pool`.
template <typename T>
cudaError_t pool_alloc(T** p, size_t count, cudaMemPool_t pool, cudaStream_t st) {
    void* v = nullptr;
    const cudaError_t e =
        taken(cudaMallocFromPoolAsync(&v, (count ? count : 1) * sizeof(T), pool, st));
    *p = e == cudaSuccess ? static_cast<T*>(v) : nullptr;
    return e;
}

}  // namespace pvs
