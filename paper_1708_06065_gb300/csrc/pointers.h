// pointers.h -- what the memory behind a caller's pointer is.
#pragma once

#include <cuda_runtime_api.h>
#include <stdint.h>

namespace lair {

inline bool pointer_attributes(const void *p, cudaPointerAttributes *a) {
    if (cudaPointerGetAttributes(a, p) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

// true for device (or managed) memory
inline bool is_device_ptr(const void *p) {
    cudaPointerAttributes a;
    return pointer_attributes(p, &a) && (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged);
}

// true for a vector that kernels on the current device read and write where it is: in this device's memory and on a
// double's boundary. What cudaMemcpyAsync takes besides (another GPU's memory, managed memory, any byte address) goes
// through a copy.
inline bool kernels_take(const double *p) {
    cudaPointerAttributes a;
    int dev = -1;
    if (reinterpret_cast<uintptr_t>(p) % alignof(double) != 0 || !pointer_attributes(p, &a)) return false;
    return a.type == cudaMemoryTypeDevice && cudaGetDevice(&dev) == cudaSuccess && a.device == dev;
}

}  // namespace lair
