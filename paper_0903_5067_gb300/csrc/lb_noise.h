// The double-precision noise tables of the current device, filled (lb_noise.cu).  Throws LbError.
#pragma once
#include "philox.cuh"

namespace gblb {
NoiseTab noise_tables();
}
