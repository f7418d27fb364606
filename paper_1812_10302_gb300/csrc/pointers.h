// pointers.h -- where an array argument lies.
#pragma once

#include <cuda_runtime_api.h>

namespace dtws {

// Whether kernels on the current device may read p where it is: its own memory,
// or managed memory.  (Another device's is copied: peer access is the
// caller's to grant, and is not assumed.)
inline bool readable_in_place(const void *p) {
    cudaPointerAttributes at;
    int device = 0;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess || cudaGetDevice(&device) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == device);
}

}  // namespace dtws
