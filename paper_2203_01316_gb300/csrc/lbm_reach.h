// Which caller's buffers a kernel may touch.
#pragma once

#include <cuda_runtime_api.h>

namespace lbmd {

// whether a kernel on `device` may read and write memory of these attributes
// itself.  Memory of another GPU is mapped there only if the program enabled
// peer access, and host memory only if it was registered, so those are left to
// cudaMemcpyAsync, which serves any of them.
inline bool kernel_reaches(const cudaPointerAttributes& a, int device) {
    return (a.type == cudaMemoryTypeDevice && a.device == device) || a.type == cudaMemoryTypeManaged;
}

}  // namespace lbmd
