// Where a caller's array lies (host code only).
#pragma once
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

namespace sph {

// Whether p is memory of the current device, aligned for elements of `align`
// bytes: a kernel may read or write it in place of a staging copy.  Host,
// managed and peer memory and addresses that only a copy can take (an array
// behind an odd number of 4-byte words in one buffer) are staged.
inline bool on_this_device(const void* p, size_t align) {
    cudaPointerAttributes at{};
    int dev = -1;
    if (!p || reinterpret_cast<uintptr_t>(p) % align != 0) return false;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice && at.device == dev;
}

// The same for an array of T.
template <typename T>
inline bool on_this_device(const T* p) {
    return on_this_device(p, alignof(T));
}

}  // namespace sph
