// Where a kernel on one device finds a caller's array (host code only).
#pragma once

#include <cuda_runtime_api.h>

namespace pic {

// The address for kernels on `device`, from the pointer's attributes: its own device
// memory, managed memory, or host memory that is pinned and mapped (kernels then read or
// write it over the host link directly, at the link's rate); null for pageable host
// memory and for another device's memory, both of which copies reach.
inline void *kernel_address(const cudaPointerAttributes &a, int device) {
  if (a.type == cudaMemoryTypeManaged || a.type == cudaMemoryTypeHost) return a.devicePointer;
  return a.type == cudaMemoryTypeDevice && a.device == device ? a.devicePointer : nullptr;
}

}  // namespace pic
