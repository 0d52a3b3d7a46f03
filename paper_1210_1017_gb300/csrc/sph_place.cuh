// Where a caller's array lies (host code only).
#pragma once
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

namespace sph {

// Whether [p, p + bytes) lies in one allocation.  A copy refuses an array that
// reaches past its allocation with an error; a kernel would fault.
inline bool in_one_allocation(const void* p, size_t bytes) {
    using Range = CUresult (*)(CUdeviceptr*, size_t*, CUdeviceptr);
    static const Range range = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &fn, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        return reinterpret_cast<Range>(fn);
    }();
    CUdeviceptr base = 0;
    size_t size = 0;
    const CUdeviceptr at = reinterpret_cast<uintptr_t>(p);
    return range && range(&base, &size, at) == CUDA_SUCCESS && at >= base && size >= bytes &&
           at - base <= size - bytes;
}

// Whether the `bytes` at p are memory of the current device, aligned for
// elements of `align` bytes: a kernel may read or write them in place of a
// staging copy.  Host, managed and peer memory and addresses that only a copy
// can take (an array behind an odd number of 4-byte words in one buffer) are
// staged, and so is what the copy refuses.
inline bool on_this_device(const void* p, size_t bytes, size_t align) {
    cudaPointerAttributes at{};
    int dev = -1;
    if (!p || reinterpret_cast<uintptr_t>(p) % align != 0) return false;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice && at.device == dev && in_one_allocation(p, bytes);
}

// The same for an array of n elements.
template <typename T>
inline bool on_this_device(const T* p, size_t n) {
    return on_this_device(p, n * sizeof(T), alignof(T));
}

}  // namespace sph
