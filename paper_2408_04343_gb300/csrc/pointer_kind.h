// Where a caller's pointer may be used.  Decisions on the attributes alone,
// checked on the CPU.
#pragma once

#include <cuda_runtime_api.h>

namespace snp {

inline bool is_device_memory(const cudaPointerAttributes& a) {
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Memory that kernels on device `dev` may read in place.  Another device's is
// mapped here only with peer access; a copy (cudaMemcpyDefault) reaches it
// either way.
inline bool readable_in_place(const cudaPointerAttributes& a, int dev) {
    return is_device_memory(a) && a.device == dev;
}

}  // namespace snp
