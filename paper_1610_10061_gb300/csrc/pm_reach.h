// Whether a kernel on `device` may store to an output of the caller by the
// 16-byte and halfword stores of the library's copies: memory of that device
// or managed memory, at an even address.  Other outputs (host memory, another
// GPU's) take the runtime's copies, which reach them.
#pragma once

#include <cuda_runtime_api.h>

#include <cstdint>

inline bool pm_kernel_may_store(const cudaPointerAttributes &a, const void *out, int device)
{
    const bool near = a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == device);
    return near && (reinterpret_cast<uintptr_t>(out) & 1u) == 0;
}
