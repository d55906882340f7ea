// Kernels that run in clusters of any size.
#pragma once
#include <driver_types.h>

namespace gblb {

// launch(size) in clusters of `size` blocks, in fewer where the device has no place for that many (a
// part of a GPU, other groups of SMs): the largest portable size, 8, then halves.  Any other
// error is the caller's.
template <class Launch>
cudaError_t launch_in_clusters(int size, Launch&& launch) {
  for (;;) {
    const cudaError_t e = launch(size);
    const bool no_place = e == cudaErrorInvalidClusterSize || e == cudaErrorLaunchOutOfResources;
    if (!no_place || size == 1) return e;
    size = size > 8 ? 8 : size / 2;
  }
}

}  // namespace gblb
