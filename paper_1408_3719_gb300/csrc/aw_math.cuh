// Device arithmetic of the sweep kernels on an FP64 pipe that takes one warp
// instruction per 16 SM cycles (64 per sub-partition): reciprocals from the
// hardware's approximation, and sums of FP64 data with small integer weights
// taken exactly on the FP32 pipe.
#pragma once
#include <cuda_runtime.h>

namespace aw {

// 1 / x by Householder's third-order iteration y (1 + e + e^2), e = 1 - x y,
// from the hardware approximation (relative error 2^-20 at worst, so e^3 is
// below 2^-60): within 1 ulp of the quotient for normal x and 1/x.  NaN where
// x is 0, infinite or subnormal (1.0 / x: infinity or 0).  Three FP64
// instructions: 50 SM cycles per warp, against 86 for 1.0 / x.
__device__ __forceinline__ double rcp3(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// x > 0 (false for NaN) without an FP64 compare
__device__ __forceinline__ bool is_positive(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000LL;
}

__device__ __forceinline__ int exponent_bits(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// The three 18-bit limbs (as exact floats; the top one signed) of x rounded
// to a multiple of 2^(E - 1022 - 54), E >= the exponent bits of x: |x| is
// below 2^(E - 1022), so the integer is below 2^54 in size and its rounding
// error is at most half an ulp of the largest number with the exponent E.
__device__ __forceinline__ float4 limbs18(double x, int E) {
  const int hi = __double2hiint(x);
  const int ex = (hi >> 20) & 0x7ff;
  unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xfffff) | (ex ? 0x100000 : 0)) << 32) |
                         (unsigned)__double2loint(x);  // 53 bits
  m <<= 1;
  const int sh = min(E - max(ex, 1), 60);
  m = (m + ((1ull << sh) >> 1)) >> sh;
  const long long q = hi < 0 ? -(long long)m : (long long)m;
  // integers below 2^22 become floats through the mantissa of 2^23 (3 * 2^22 for signed ones)
  float4 f;
  f.x = __int_as_float(0x4b400000 + (int)(q >> 36)) - 12582912.0f;
  f.y = __int_as_float(0x4b000000 | ((int)(q >> 18) & 0x3ffff)) - 8388608.0f;
  f.z = __int_as_float(0x4b000000 | ((int)q & 0x3ffff)) - 8388608.0f;
  f.w = 0.0f;
  return f;
}

// 2^(E - 1022 - 54), the unit of limbs18; NaN for the exponent of infinities
// and NaN, so that a sum over non-finite data is NaN
__device__ __forceinline__ double limb_unit(int E) {
  return E >= 0x7ff ? __longlong_as_double(0x7ff8000000000000LL) : __hiloint2double((E - 53) << 20, 0);
}

// sum of limbs back to one double (in units of limb_unit): exact below 2^53,
// one rounding above.  Each limb sum is an integer below 2^24.
__device__ __forceinline__ double join18(float s2, float s1, float s0) {
  const long long q = ((long long)__float2int_rn(s2) << 36) + ((long long)__float2int_rn(s1) << 18) +
                      (long long)__float2int_rn(s0);
  return (double)q;
}

}  // namespace aw
