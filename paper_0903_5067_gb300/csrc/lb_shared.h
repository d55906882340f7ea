// Dynamic shared memory beyond the 48 KB every kernel may use without asking.
#pragma once
#include <cuda_runtime.h>

namespace gblb {

// Allow a kernel, on the current device, all the shared memory a block can have beside its static
// part.  The attribute belongs to the kernel, not to an object or a launch: set to what one object
// needs, it would refuse the launches of an earlier, larger one, or of another thread between its
// setting and its launch.  Always set to the same value, it does neither.
inline cudaError_t allow_all_shared(const void* kernel) {
  cudaFuncAttributes a;
  int dev = 0, most = 0;
  cudaError_t e = cudaFuncGetAttributes(&a, kernel);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
  return e;
}

}  // namespace gblb
