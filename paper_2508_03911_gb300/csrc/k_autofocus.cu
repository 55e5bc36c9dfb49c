// k_autofocus.cu -- the Tamura coefficient of the autofocus sweep from per-frame amplitude
// sums.
//
// The plain z-sweep the network replaces: for every distance z_j, the angular
// spectrum propagation of the mean-removed hologram (Sec. III-B.1's ASP with the
// DC bin of the transfer function set to zero) and the Tamura coefficient
// sqrt(sigma / mu) of the amplitude |U| over the frame.
#include "hv_internal.h"

namespace hv {

namespace {

// metric[i] = sqrt(sigma / mu) of frame-and-distance i from (sum |u|, sum |u|^2)
// over P pixels; 0 when mu = 0.
__global__ void k_tamura_finish(const double* acc, uint32_t count, double P, float* metric) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const double mu = acc[2 * i] / P;
    const double var = acc[2 * i + 1] / P - mu * mu;
    const double sigma = var > 0.0 ? sqrt(var) : 0.0;
    metric[i] = mu > 0.0 ? float(sqrt(sigma / mu)) : 0.f;
  }
}

}  // namespace

cudaError_t launch_tamura_finish(const double* acc, uint32_t count, uint32_t pixels, float* metric, cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const uint32_t blocks = (count + 255) / 256;
  k_tamura_finish<<<blocks < 1024 ? blocks : 1024, 256, 0, s>>>(acc, count, double(pixels), metric);
  return cudaGetLastError();
}

}  // namespace hv
