// quotient.h -- the normalised moments M1 / M0 and sqrt(M2 / M0) of float32 moments, as float64
// gives them. Float64 instructions run at 1/64 of the float32 rate, and one lane in 4 to 16
// writes: in float64 the two took 0.1 ms per window of 1024 x 512.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace hv {

// float(double(a) / double(b)): the float32 quotient is the same number, since float64 keeps
// more than twice float32's digits and two bits (results below the normal range apart, which
// float64 rounds twice).
__host__ __device__ __forceinline__ float quotient(float a, float b) { return a / b; }

// float(sqrt(double(a) / double(b))) for a >= 0, b > 0: the quotient as a float32 pair (its
// remainder exact by fma), one Newton step of the root on the pair. The step's length is right
// to a few times 2^-24; where a millionth more or less of it rounds to another float32 (one in a
// million), and outside the range where the pair holds, the float64 form (taking the step
// unchecked, 7 of 3e8 pairs came out one unit off).
__host__ __device__ __forceinline__ float root_of_quotient(float a, float b) {
  const float q = a / b;
  if (a > 1e-25f && b > 1e-25f && b < 1e25f && q > 1e-25f && q < 1e25f) {
    const float lo = fmaf(-q, b, a) / b;
    const float s = sqrtf(q);
    const float h = 0.5f * (1.f / s), r = fmaf(-s, s, q) + lo;
    const float most = fmaf(h, r * 1.00000095367431640625f, s), least = fmaf(h, r * 0.99999904632568359375f, s);
    if (most == least) return most;
  }
  const double r = double(a) / double(b);
  return float(sqrt(r > 0.0 ? r : 0.0));
}

}  // namespace hv
