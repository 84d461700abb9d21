// Whether a kernel may read a caller's array where it lies (cliffs_set_initial,
// cliffs_depth_filter_noalloc) or the copy engine has to bring it over first.
#pragma once
#include <cuda_runtime_api.h>
#include <stdint.h>

namespace cliffs {

// type and owner: what cudaPointerGetAttributes says of the address p; current: the current
// device; size: of an element. The copy engine takes memory of any device and any byte address;
// a load in a kernel faults on another device's memory (no peer access) and on an address that
// is not a multiple of the element size. Managed memory is left to the copy engine too.
inline bool kernel_may_read(cudaMemoryType type, int owner, int current, const void* p, size_t size) {
    return type == cudaMemoryTypeDevice && owner == current && reinterpret_cast<uintptr_t>(p) % size == 0;
}

template <class T>
inline bool kernel_may_read(const T* p) {
    cudaPointerAttributes at;
    int dev = -1;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) { cudaGetLastError(); return false; }
    return cudaGetDevice(&dev) == cudaSuccess && kernel_may_read(at.type, at.device, dev, p, sizeof(T));
}

}  // namespace cliffs
