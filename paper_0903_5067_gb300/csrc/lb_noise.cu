// The radii and angles of the double-precision fluid noise (NoiseTab), once per device.
//
// The tables are constants, the same for every context, so they are file-scope device arrays (16 MiB
// and 32 KiB) that a GPU holds from the first double-precision context on it until the process
// exits; with them in each context's workspace, a box of L = 32 would need 27 instead of 10 MB.
#include <cuda_runtime.h>

#include "lb_engine.h"
#include "lb_noise.h"

namespace gblb {
namespace {

constexpr unsigned kFillBlocks = 304;  // two per SM
constexpr unsigned kFilled = 0x5a5a5a5au;
struct Tables {
  double radius[kRadii];
  double2 angle[kAngles];
  unsigned filled[kFillBlocks];  // kFilled once the block's share holds its values
};
__device__ __align__(256) Tables g_tab;

// 0.15 ms the first time on a device: a logarithm and a square root per radius; then nothing to do.  A
// block looks at, and sets behind its writes, the mark of its own share.
__global__ void fill_noise_tables() {
  const bool filled = threadIdx.x == 0 && *(volatile unsigned*)&g_tab.filled[blockIdx.x] == kFilled;
  if (__syncthreads_or(filled)) return;
  for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < kRadii; k += gridDim.x * blockDim.x) {
    g_tab.radius[k] = sqrt(-2.0 * log(((double)k + 0.5) * 0x1p-21));
    if (k < kAngles) {
      double s, c;
      sincospi(2.0 * (((double)k + 0.5) * 0x1p-11) - 1.0, &s, &c);
      g_tab.angle[k] = make_double2(c, s);
    }
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *(volatile unsigned*)&g_tab.filled[blockIdx.x] = kFilled;
}

// the calling thread's capture mode relaxed: another stream that is being captured is not disturbed
// by the loading of this file's device code
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cuda_check(cudaThreadExchangeStreamCaptureMode(&mode), "capture mode"); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

}  // namespace

// Whether they are filled is read on the device, not remembered here: a device that was reset has lost
// them.  One kernel on the caller's stream and no wait: what follows it there finds the tables
// filled.  Streams that come at the same time may fill a share twice, with the same values.  (A look
// at a mark from the host, on a stream made for it, made a context of L = 16 start in 61 us instead of
// the 42 it took without tables; now 39.)
NoiseTab noise_tables(cudaStream_t s) {
  const RelaxedCapture relaxed;
  void* p = nullptr;
  cuda_check(cudaGetSymbolAddress(&p, g_tab), "noise tables");
  fill_noise_tables<<<kFillBlocks, 256, 0, s>>>();
  cuda_check(cudaGetLastError(), "noise tables");
  const Tables* t = static_cast<const Tables*>(p);
  return NoiseTab{t->radius, t->angle};
}

}  // namespace gblb
