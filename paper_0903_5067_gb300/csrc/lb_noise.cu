// The radii and angles of the double-precision fluid noise (NoiseTab), once per device.
//
// The tables are constants, the same for every context, so they are file-scope device arrays (16 MiB
// and 32 KiB) that a GPU holds from the first double-precision context on it until the process
// exits; with them in each context's workspace, a box of L = 32 would need 27 instead of 10 MB.
#include <cuda_runtime.h>

#include <mutex>

#include "lb_engine.h"
#include "lb_noise.h"

namespace gblb {
namespace {

__device__ __align__(256) double g_radius[kRadii];
__device__ __align__(256) double2 g_angle[kAngles];
__device__ double g_filled;  // kFilled once the tables hold their values
constexpr double kFilled = 0x1.5a5a5p0;

// 0.15 ms: a logarithm and a square root per radius
__global__ void fill_noise_tables() {
  for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < kRadii; k += gridDim.x * blockDim.x) {
    g_radius[k] = sqrt(-2.0 * log(((double)k + 0.5) * 0x1p-21));
    if (k < kAngles) {
      double s, c;
      sincospi(2.0 * (((double)k + 0.5) * 0x1p-11) - 1.0, &s, &c);
      g_angle[k] = make_double2(c, s);
    }
  }
}
__global__ void mark_filled() { g_filled = kFilled; }

// a stream of its own, and the calling thread's capture mode relaxed: another stream that is being
// captured neither takes part nor is disturbed
struct Stream {
  cudaStream_t s = nullptr;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  Stream() {
    cuda_check(cudaThreadExchangeStreamCaptureMode(&mode), "capture mode");
    const cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e != cudaSuccess) cudaThreadExchangeStreamCaptureMode(&mode);
    cuda_check(e, "noise stream");
  }
  ~Stream() {
    cudaStreamDestroy(s);
    cudaThreadExchangeStreamCaptureMode(&mode);
  }
};

}  // namespace

// Whether they are filled is read from the device, not remembered: a device that was reset has lost
// them.  The caller may use them on any stream: the fill has completed when this returns.
NoiseTab noise_tables() {
  static std::mutex mu;
  const std::lock_guard<std::mutex> lock(mu);
  void *radius = nullptr, *angle = nullptr, *filled = nullptr;
  cuda_check(cudaGetSymbolAddress(&radius, g_radius), "noise radii");
  cuda_check(cudaGetSymbolAddress(&angle, g_angle), "noise angles");
  cuda_check(cudaGetSymbolAddress(&filled, g_filled), "noise mark");
  Stream st;
  double mark = 0.0;
  cuda_check(cudaMemcpyAsync(&mark, filled, sizeof(mark), cudaMemcpyDeviceToHost, st.s), "noise mark");
  cuda_check(cudaStreamSynchronize(st.s), "noise mark");
  if (mark != kFilled) {
    fill_noise_tables<<<1216, 256, 0, st.s>>>();
    cuda_check(cudaGetLastError(), "noise tables");
    mark_filled<<<1, 1, 0, st.s>>>();
    cuda_check(cudaGetLastError(), "noise mark");
    cuda_check(cudaStreamSynchronize(st.s), "noise tables");
  }
  return NoiseTab{static_cast<const double*>(radius), static_cast<const double2*>(angle)};
}

}  // namespace gblb
