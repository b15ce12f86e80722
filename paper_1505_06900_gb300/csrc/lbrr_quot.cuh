// What the kernels for runs of updates (lbrr_run2.cu, lbrr_run2m.cu, lbrr_run3.cu)
// use to form j / rho as the division of a single update rounds it, without a
// division for each component.
#pragma once

#include <cuda_runtime.h>

namespace lbrr {

__device__ __forceinline__ float approx_reciprocal(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// The correctly rounded -1 / x: one Newton step from the hardware's
// approximation. Compared with __frcp_rn for every significand in binades from
// 2^-67 to 2^67, the one of all ones included (rho = 1 - 2^-24), where the step
// from the farther neighbour of 1 / x would not get there.
__device__ __forceinline__ float minus_reciprocal(float x) {
  const float r = approx_reciprocal(-x);
  return __fmaf_rn(__fmaf_rn(x, r, 1.0f), r, r);
}

// The correction does not give the correct rounding where the remainder need not
// be a number of FP32, for a quotient u next to zero (rho is zero or 2^-24 at
// least), nor where there is no reciprocal (u is NaN). Division then; a momentum
// of zero needs none, so the smallest |u| of a cell is looked at first.
constexpr float kLeastQuotient = 0x1p-78f;
__device__ __forceinline__ bool needs_division(float j, float u) {
  return !(fabsf(u) >= kLeastQuotient) && j != 0.0f;
}

}  // namespace lbrr
