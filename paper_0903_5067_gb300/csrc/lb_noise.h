// The double-precision noise tables of the current device, filled for what follows on s (lb_noise.cu).
// Throws LbError.
#pragma once
#include <cuda_runtime.h>

#include "philox.cuh"

namespace gblb {
NoiseTab noise_tables(cudaStream_t s);
}
