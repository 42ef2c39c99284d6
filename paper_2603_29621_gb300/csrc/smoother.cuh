// One smoother update, shared by every kernel that applies it: explicit fused operations, so that the
// update rounds alike wherever it is fused.
#pragma once
#include <cuda_runtime.h>

namespace mfns {

// a product that no later addition is fused into
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// new direction c1 d + c2 dinv res; c1 = 0 (a first step): d is not used, it may be unset
template <typename T>
__device__ __forceinline__ T smoother_direction(T c1, T c2, T d, T dinv, T res) {
  const T s = mul_rn(mul_rn(c2, dinv), res);
  return c1 != T(0) ? fma(c1, d, s) : s;
}

}  // namespace mfns
