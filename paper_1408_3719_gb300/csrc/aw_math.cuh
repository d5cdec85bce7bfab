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

// sqrt(x) = g (1 - e)^(-1/2), g = x y, e = 1 - g y, from the hardware
// approximation y of 1 / sqrt(x) (relative error 2^-20 at worst) and the
// binomial series to e^2: within 1 ulp for normal x.  Five FP64 instructions:
// 82 SM cycles per warp, against 143 for sqrt(x).  0 for zeros and subnormal x
// (below 1.5e-154), NaN for negative and infinite x.
__device__ __forceinline__ double sqrt5(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y, e = fma(-g, y, 1.0);
  const double s = fma(g * e, fma(0.375, e, 0.5), g);
  return (__double2hiint(x) & 0x7ff00000) == 0 ? 0.0 : s;
}
// 1 / sqrt(x), likewise (NaN for zeros and subnormal x)
__device__ __forceinline__ double rsqrt5(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// x as an integer of 2^(E - 1022 - BITS), rounded half away from zero, for E
// >= the exponent bits of x: below 2^BITS in size (BITS 53..62).
template <int BITS>
__device__ __forceinline__ long long fixed_point(double x, int E) {
  const int hi = __double2hiint(x);
  const int ex = (hi >> 20) & 0x7ff;
  unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xfffff) | (ex ? 0x100000 : 0)) << 32) |
                         (unsigned)__double2loint(x);  // 53 bits
  m <<= BITS - 53;
  const int sh = min(E - max(ex, 1), 63);
  m = (m + ((1ull << sh) >> 1)) >> sh;
  return hi < 0 ? -(long long)m : (long long)m;
}

// The three 18-bit limbs (as exact floats; the top one signed) of x rounded
// to a multiple of 2^(E - 1022 - 54), E >= the exponent bits of x: |x| is
// below 2^(E - 1022), so the integer is below 2^54 in size and its rounding
// error is at most half an ulp of the largest number with the exponent E.
__device__ __forceinline__ float4 limbs18(double x, int E) {
  const long long q = fixed_point<54>(x, E);
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

// (double)q for |q| <= 2^62 on the integer pipes, the same to the bit: the
// conversion instruction takes the FP64 pipe's 16 SM cycles, these two dozen
// about 10, though more time from end to end
__device__ __forceinline__ double int_to_double(long long q) {
  const unsigned long long a = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << ((lz - 1) & 63);  // 2^62 <= m < 2^63
  const unsigned long long r = (m + 0x1ff + ((m >> 10) & 1)) >> 10;  // 53 bits, or 2^53
  const unsigned long long b = ((unsigned long long)(unsigned)(1085 - lz) << 52) + r;
  return __longlong_as_double(a ? (long long)(b | (q < 0 ? 0x8000000000000000ull : 0ull)) : 0ll);
}

// sum of limbs back to one double (in units of limb_unit): exact below 2^53,
// one rounding above.  Each limb sum is an integer below 2^24.
template <bool INT>
__device__ __forceinline__ double join18(float s2, float s1, float s0) {
  const long long q = ((long long)__float2int_rn(s2) << 36) + ((long long)__float2int_rn(s1) << 18) +
                      (long long)__float2int_rn(s0);
  return INT ? int_to_double(q) : (double)q;
}

// A 57-bit integer in two limbs, q = h 2^28 + l with -2^27 <= l < 2^27: sums
// of up to 31 products of two such numbers as h h and h l + l h in 64-bit
// integers (the dropped l l are below 2^-58 of the largest product).
__device__ __forceinline__ int2 limbs28(long long q) {
  const int h = (int)((q + (1ll << 27)) >> 28);
  return make_int2(h, (int)(q - ((long long)h << 28)));
}
__device__ __forceinline__ void dot28(long long& hh, long long& hl, int2 a, int2 b) {
  hh += (long long)a.x * b.x;
  hl += (long long)a.x * b.y;
  hl += (long long)a.y * b.x;
}

// Unevaluated sums of two floats (48 bits), after Dekker (1971) and Knuth's
// two-sum: an FP64-like accumulation on the FP32 pipe.
struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 f2_norm(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
// a - x y; the result is not normalised
__device__ __forceinline__ F2 f2_sub_mul(F2 a, F2 x, F2 y) {
  const float p = __fmul_rn(x.h, y.h);
  const float e = __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.l, __fmaf_rn(x.h, y.h, -p)));
  const float s = __fsub_rn(a.h, p), t = __fsub_rn(s, a.h);
  const float err = __fsub_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fadd_rn(p, t));
  return {s, __fadd_rn(a.l, __fsub_rn(err, e))};
}
// a + b, normalised
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
  const float err = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
  return f2_norm(s, __fadd_rn(err, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 f2_mul(F2 x, F2 y) {
  const float p = __fmul_rn(x.h, y.h);
  return f2_norm(p, __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.l, __fmaf_rn(x.h, y.h, -p))));
}
// 1 / sqrt(d) from the hardware approximation and two terms of the binomial
// series; not finite for d <= 0
__device__ __forceinline__ F2 f2_rsqrt(F2 d) {
  const float y = rsqrtf(d.h), p = __fmul_rn(y, y), e = __fmaf_rn(y, y, -p);
  const float r = __fmaf_rn(-d.l, p, __fmaf_rn(-d.h, e, __fmaf_rn(-d.h, p, 1.0f)));
  return f2_norm(y, __fmul_rn(__fmul_rn(y, r), __fmaf_rn(0.375f, r, 0.5f)));
}
// hh 2^56 + hl 2^28 (sums of dot28) in units of 2^56: 48 bits
__device__ __forceinline__ F2 f2_of_dot(long long hh, long long hl) {
  const long long q = hh + (hl >> 28);
  const float f3 = (float)(int)(q >> 40);
  const float f2 = __int_as_float(0x4b000000 | ((int)(q >> 20) & 0xfffff)) - 8388608.0f;
  const float f1 = __int_as_float(0x4b000000 | ((int)q & 0xfffff)) - 8388608.0f;
  const float f0 = (float)((int)hl & 0xfffffff);
  return f2_add(f2_norm(f3 * 1099511627776.0f, f2 * 1048576.0f), f2_norm(f1, f0 * 0x1p-28f));
}
// a 2^k as an integer of 2^-57 (|a| 2^k below 1/2)
__device__ __forceinline__ long long f2_fixed57(F2 a, float pow2_28k) {  // 2^(28 + k)
  const float t = a.h * pow2_28k;
  const int i = __float2int_rn(t);
  const float r = __fadd_rn(__fsub_rn(t, (float)i), a.l * pow2_28k);
  return ((long long)i << 29) + (long long)__float2int_rn(r * 536870912.0f);
}

}  // namespace aw
