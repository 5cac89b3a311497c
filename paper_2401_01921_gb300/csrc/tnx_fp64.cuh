// FP64 values handled on the integer units.  A warp's FP64 instruction occupies its SM
// quarter's FP64 unit for 64 cycles on this part, however few lanes need it; integer
// instructions take 2.
#pragma once

#include <cuda_runtime.h>

namespace tnx_fp64 {

__device__ __forceinline__ int expo(int hi) { return (hi >> 20) & 0x7FF; }   // biased exponent
__device__ __forceinline__ float mant(double x) {                             // |mantissa| in [1, 2), 23 bits
  return __int_as_float(0x3F800000 | ((__double2hiint(x) & 0xFFFFF) << 3) |
                        (int)((unsigned)__double2loint(x) >> 29));
}

// x * 2^k rounded to an integer (0 when x is zero or subnormal or the result is
// below 1/2 or, for an x that is not finite, above 2^62).
__device__ __forceinline__ long long scaled_int(double x, int k) {
  const int hi = __double2hiint(x), e = expo(hi) - 1023 + k;   // |x| 2^k in [2^e, 2^(e+1))
  if (expo(hi) == 0 || e < -1 || e > 61) return 0;
  const long long m = ((long long)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(x);   // 53 bits
  const long long v = e >= 52 ? m << (e - 52) : ((m >> (51 - e)) + 1) >> 1;
  return hi < 0 ? -v : v;
}

// Sum over the warp of |v| <= 2^60 in total: limbs of 21, 21 and 20 bits.
__device__ __forceinline__ long long warp_sum_int(long long v) {
  const int lo = __reduce_add_sync(0xffffffffu, (int)(v & 0x1FFFFF));
  const int mid = __reduce_add_sync(0xffffffffu, (int)((v >> 21) & 0x1FFFFF));
  const int hi = __reduce_add_sync(0xffffffffu, (int)(v >> 42));
  return ((long long)hi << 42) + ((long long)mid << 21) + lo;
}

// Sum of a double over the warp as v 2^-k: the lanes' values rounded to units of 2^-54
// of the largest (it lies below 2^(top - 1022), so 32 of them in units of 2^-k stay
// below 2^60).
__device__ __forceinline__ long long warp_sum_scaled(double x, int& k) {
  const int top = __reduce_max_sync(0xffffffffu, expo(__double2hiint(x)));
  k = 55 - (top - 1022);
  return warp_sum_int(scaled_int(x, k));
}

// x * 2^-k for a normal or zero x (0 below the normal range, an infinity above it)
__device__ __forceinline__ double shift_down(double x, int k) {
  const int hi = __double2hiint(x), e = expo(hi) - k;
  if (expo(hi) == 0 || e <= 0) return 0.0;
  if (e >= 2047) return __hiloint2double((hi & 0x80000000) | 0x7FF00000, 0);
  return __hiloint2double((hi & 0x800FFFFF) | (e << 20), __double2loint(x));
}

__device__ __forceinline__ bool is_finite(double x) { return expo(__double2hiint(x)) != 2047; }

// Sum of a double over the warp, in every lane (NaN when a value is not finite, an infinity
// when the sum of finite values is not; subnormal values count as zero).
__device__ __forceinline__ double warp_sum_double(double x) {
  int k;
  const long long v = warp_sum_scaled(x, k);
  return k == 55 - (2047 - 1022) ? __longlong_as_double(0x7FF8000000000000ll) : shift_down((double)v, k);
}

}  // namespace tnx_fp64
