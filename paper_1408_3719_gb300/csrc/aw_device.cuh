// Small device functions of the sweep kernels (aw_kernels.cu and aw_plain.cu).
#pragma once
#include "aw_internal.h"

namespace aw {

__device__ __forceinline__ double area6(const double* X) {
  return 0.5 * ((X[2] - X[0]) * (X[5] - X[1]) - (X[3] - X[1]) * (X[4] - X[0]));
}

__device__ __forceinline__ void set_error(Counters* cnt, int code, int elem) {
  if (atomicCAS(&cnt->err_code, 0, code) == 0) cnt->err_elem = elem;
}

__device__ __forceinline__ double pressure(const Tab& T, const double* q) {
  return (T.gamma - 1.0) * (q[3] - 0.5 * (q[1] * q[1] + q[2] * q[2]) / q[0]);
}

}  // namespace aw
