// Which memory elitekv_copy takes (apart from the runtime calls, so that the rule can be looked at without
// a device).
#pragma once

#include <cuda_runtime_api.h>

// Kernels of `device` can address p: pinned host memory or managed memory under the same address, or memory
// of this device.  Another device's memory is not taken: whether it may be addressed depends on peer access.
inline bool ekv_addressable(const cudaPointerAttributes& at, const void* p, int device) {
  return at.type != cudaMemoryTypeUnregistered && at.devicePointer == p && (at.type != cudaMemoryTypeDevice || at.device == device);
}
