// Reciprocals of positive numbers in [2^-120, 2^120] (the launch rules keep eps within 2^+-100).
#pragma once

#include <cuda_runtime.h>

namespace gks {

// FP32: the hardware reciprocal (1 ulp), without the scaling that __fdividef adds for subnormal and
// huge divisors (6 instructions a value).
__device__ __forceinline__ float rcp_normal(float s) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s));
  return r;
}

// FP64: one third-order (Chebyshev) step r (1 + e + e^2), e = 1 - x r, from the FP32 reciprocal of x
// rounded down to FP32.  |e| < 2^-21, so e^3 is far below an ulp and the result is within 0.51 ulp.
// Three FP64 operations instead of the division's 9 (the FP64 pipe takes 64 cycles for each); the
// conversions are integer operations.
__device__ __forceinline__ double rcp_normal(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const float f = __int_as_float(((hi - (896 << 20)) << 3) | (int)((unsigned)lo >> 29));
  const int b = __float_as_int(rcp_normal(f));
  const double r = __hiloint2double((b >> 3) + (896 << 20), b << 29);
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace gks
