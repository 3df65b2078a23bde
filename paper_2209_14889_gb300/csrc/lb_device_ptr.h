// lb_device_ptr.h -- whether a kernel may write a buffer that a caller calls device memory.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace vlb {

// [p, p + bytes) begins and ends in memory of the current device and holds aligned 4-byte values.  A
// copy refuses or handles what is not (host memory, another device's, an odd address); a kernel
// that wrote there would fault.
inline bool device_floats(const void* p, size_t bytes)
{
    int dev = -1;
    if (bytes == 0 || (reinterpret_cast<uintptr_t>(p) & 3) || cudaGetDevice(&dev) != cudaSuccess) return false;
    const char* ends[2] = {static_cast<const char*>(p), static_cast<const char*>(p) + bytes - 1};
    for (const char* e : ends) {
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, e) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (at.type != cudaMemoryTypeDevice || at.device != dev) return false;
    }
    return true;
}

}  // namespace vlb
