// What the two summary builders share: the FP4 quantiser's arithmetic.
#pragma once

#include "common.cuh"

namespace cobs {

// code = sign bit of x, nearest E2M1 magnitude to |x| / scale with ties to the even mantissa bit.
__device__ __forceinline__ uint32_t e2m1_encode(float x, float scale) {
  const float t = __fdiv_rn(fabsf(x), scale);
  uint32_t m = 0;
  m += (t > 0.25f);
  m += (t >= 0.75f);
  m += (t > 1.25f);
  m += (t >= 1.75f);
  m += (t > 2.5f);
  m += (t >= 3.5f);
  m += (t > 5.0f);
  return (signbit(x) ? 8u : 0u) | m;
}

// scale of a factor row whose largest magnitude is a
__device__ __forceinline__ float fp4_scale(float a, int scale_dtype) {
  float scale = __fdiv_rn(a, 6.0f);
  if (scale_dtype == COBS_SCALE_FP16) scale = __half2float(__float2half_rn(scale));
  return scale;
}

}  // namespace cobs
