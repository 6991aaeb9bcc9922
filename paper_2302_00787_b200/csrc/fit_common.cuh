// Scalar pieces shared by the parameter-fit kernels.
#pragma once
#include "common.cuh"

namespace {

// Lemma A.1 in the cancellation-free form that follows from its proof:
// 1 - 8A = (2 phi + 1 + s)/2 with s = sqrt((2 phi + 1)^2 + 8 phi).
__device__ __forceinline__ double lemma_a1(double phi) {
  double s = sqrt((2.0 * phi + 1.0) * (2.0 * phi + 1.0) + 8.0 * phi);
  return -(2.0 * phi + (12.0 * phi + 4.0 * phi * phi) / (1.0 + s)) / 16.0;
}

// 1 / sqrt(t) and 1 / t to rounding: the 20-bit hardware estimate and two Newton steps (t normal and positive,
// resp. non-zero; no special cases).
__device__ __forceinline__ double rsqrt_fast(double t) {
  double q;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(q) : "d"(t));
  q = fma(q * 0.5, fma(-t * q, q, 1.0), q);
  return fma(q * 0.5, fma(-t * q, q, 1.0), q);
}
__device__ __forceinline__ double recip_fast(double t) {
  double q;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(q) : "d"(t));
  q = fma(q, fma(-t, q, 1.0), q);
  return fma(q, fma(-t, q, 1.0), q);
}

}  // namespace
