// Dynamic shared memory above 48 KB.
#pragma once
#include <cuda_runtime.h>

namespace gbd {

// Allows the kernel `bytes` of dynamic shared memory on the current device;
// false where that is refused.  The limit belongs to the device, so it is set
// at every launch: set once for the process, it left every device but the
// first at 48 KB.
template <class... Args>
inline bool allow_shared_memory(void (*kernel)(Args...), int bytes) {
  if (cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) ==
      cudaSuccess)
    return true;
  cudaGetLastError();   // the caller reports it
  return false;
}

}  // namespace gbd
