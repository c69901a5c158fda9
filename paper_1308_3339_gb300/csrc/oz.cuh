// FP64 operands as signed 9-bit digits and their products' sums as integers: what the FP64 form's
// near field (p2p_f64.cu, which explains the method) and M2L (m2l_f64.cu) share.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace fmmpc {

constexpr int OZ_S = 7;     // digits
constexpr int OZ_LSB = 56;  // unit 2^-56 of one offset's sum
constexpr int OZ_NONE = -(1 << 20), OZ_NAN = 1 << 20;  // exponents of an empty and of a non-finite group

// digits of X (|X| <= 2^62): X = sum_i d[i] 2^(9 (6 - i)), |d| <= 256
__device__ __forceinline__ void oz_digits(long long X, int (&d)[OZ_S]) {
#pragma unroll
  for (int i = OZ_S - 1; i > 0; --i) {
    d[i] = (int)((X + 256) & 511) - 256;
    X = (X - d[i]) >> 9;
  }
  d[0] = (int)X;
}

// Bits of |x|: those of non-negative doubles order like the values.  The biased exponent em of a group's
// largest value, at least 1: |x| < 2^(em - 1022), subnormal numbers included.
__device__ __forceinline__ unsigned long long oz_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ int oz_biased(unsigned long long mx) { return max((int)(mx >> 52), 1); }

// x as a fixed-point number below its group's exponent E = em - 1022, X = x 2^(62 - E) (0 in a non-finite
// group); l1 += |X|, rounded up
__device__ __forceinline__ long long oz_fixed(double x, int em, float &l1) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  const long long mant = (long long)((u & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull));
  const int sh = 9 - (em - max(ex, 1));
  long long X = sh >= 0 ? mant << sh : (sh > -60 ? (mant + (1ll << (-sh - 1))) >> -sh : 0);
  if (em == 0x7ff) X = 0;
  l1 += __ll2float_ru(X);
  return (u >> 63) ? -X : X;
}

// (exponent, L1 norm / 2^E rounded up) of a group
__device__ __forceinline__ int2 oz_group(unsigned long long mx, int em, float l1) {
  return make_int2(mx == 0 ? OZ_NONE : (em == 0x7ff ? OZ_NAN : em - 1022),
                   __float_as_int(l1 * (0x1p-62f * 1.00001f)));
}

// a target's bound: the sum l1 of its sources' L1 norms, in units of 2^emax, takes group v
__device__ __forceinline__ void oz_bound(int2 v, int &emax, float &l1) {
  const int e = max(emax, v.x);
  l1 = l1 * exp2f((float)max(emax - e, -200)) + __int_as_float(v.y) * exp2f((float)max(v.x - e, -200));
  emax = e;
}
// its unit 2^-lsb: the sum of the bounds stays below 2^61 (one bit for the roundings)
__device__ __forceinline__ int oz_unit(float l1) { return min(OZ_LSB, 60 - max(ilogbf(fmaxf(l1, 1.0f)), 0)); }

// the orders' sums joined in units of 2^-56: order s is in units of 2^(-9 s - 16)
__device__ __forceinline__ int oz_join_low(float v4, float v5, float v6) {
  const int s6 = __float2int_rn(v6), s5 = __float2int_rn(v5), s4 = __float2int_rn(v4);
  return s4 * 16 + ((s5 + ((s6 + 256) >> 9) + 16) >> 5);
}
__device__ __forceinline__ long long oz_join(int low, float v0, float v1, float v2, float v3) {
  long long t = (long long)low;
  t += (long long)__float2int_rn(v3) * (1 << 13);
  t += (long long)__float2int_rn(v2) * (1 << 22);
  t += (long long)__float2int_rn(v1) * (1ll << 31);
  t += (long long)__float2int_rn(v0) * (1ll << 40);
  return t;
}

static __global__ void k_oz_fill(int64_t total, int2 *__restrict__ le) {  // empty groups
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < total) le[t] = make_int2(OZ_NONE, 0);
}

}  // namespace fmmpc
