// Reciprocal roots and quotients for the selection's serial chains, where an IEEE root or division (its
// range checks and branches) is longer than what surrounds it.  Both are one Newton-Raphson step.
#pragma once
#include <cmath>
#include <cuda_runtime.h>

namespace mapk {

// 1 / sqrt(x), x > 0: the hardware estimate (at most 2 ulp off) and one Newton-Raphson step for
// f(y) = 1 / y^2 - x, y' = y + y (1 - x y^2) / 2.  Within 1 ulp (1.0f / sqrtf(x), the
// quotient of a rounded root, within 1.5); 0 for x = inf.
__device__ __forceinline__ float inv_sqrt(float x) {
  const float y = rsqrtf(x), t = x * y;
  return x < INFINITY ? fmaf(0.5f * y, fmaf(-t, y, 1.0f), y) : 0.f;
}

// a / r from the rounded reciprocal rinv = 1.0f / r: q = a rinv, then one Newton-Raphson step for
// f(q) = q r - a, the remainder exact by the fused multiply-add: within 0.51 ulp where nothing overflows
// or underflows (no difference from a / r in 2^30 random pairs).
__device__ __forceinline__ float quotient(float a, float r, float rinv) {
  const float q = a * rinv;
  return fmaf(fmaf(-q, r, a), rinv, q);
}

}  // namespace mapk
