// user_memory.cuh -- which of the caller's "device" pointers a kernel may dereference (host code only).
#pragma once
#include <cuda_runtime_api.h>
#include <stdint.h>

namespace sslbm {

// Whether a kernel on device `device` reads or writes values of `size` bytes at p directly: device
// memory of that device, at the values' alignment.  All else is left to the runtime's copies, which
// handle it or return an error -- memory of another device, and host memory that was passed as
// device memory, pageable memory among it, which a kernel may not touch.
inline bool kernel_may_use(cudaMemoryType type, int memory_device, int device, uintptr_t p, size_t size) {
  return p % size == 0 && type == cudaMemoryTypeDevice && memory_device == device;
}

}  // namespace sslbm
