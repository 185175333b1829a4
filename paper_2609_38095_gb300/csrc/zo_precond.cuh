// zo_precond.cuh -- the probe-space preconditioner of one probe (Sec. 4.1, Eqs.
// 3-4), fp64 throughout.
#pragma once

#include <cuda_runtime.h>

namespace zo {

__device__ __forceinline__ double probe_curvature(double lp, double lm, double l0, double eps) {
  return __ddiv_rn(__dadd_rn(__dsub_rn(lp, __dmul_rn(2.0, l0)), lm), __dmul_rn(eps, eps));
}

__device__ __forceinline__ double probe_weight(double r, double alpha, double lambda_reg) {
  return __ddiv_rn(1.0, fmax(lambda_reg, pow(fabs(r), alpha)));
}

__device__ __forceinline__ double central_difference(double lp, double lm, double eps) {
  return __ddiv_rn(__dsub_rn(lp, lm), __dmul_rn(2.0, eps));
}

}  // namespace zo
