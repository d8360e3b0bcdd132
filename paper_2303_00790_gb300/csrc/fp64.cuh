// FP64 helpers for kernels whose time is a chain of dependent FP64 operations.
//
// The GB300 issues an FP64 warp instruction per 64 cycles and SM sub-partition: 65 cycles from
// one dependent operation to the next, and comparisons, conversions and maxima cost the same.
// What can be done on the integer pipes is done there.
#pragma once

#include <cuda_runtime.h>

namespace kscf {

// A tree of five shuffles and additions costs ~560 cycles, all of it on the FP64 pipe's time for
// 320.  The sum is therefore formed in integers: every value is aligned to the largest
// exponent of the warp as a 58-bit integer (cut below 2^-57 of the largest value, where each
// addition of the tree rounds at 2^-53), the integers are summed exactly as three 26-bit parts
// by integer reductions, and the total is rounded to a double once.  Warps whose largest value
// is near the ends of the range (Inf, NaN and subnormal sums among them) take the tree.
__device__ __forceinline__ double warp_sum(double v) {
  const long long b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const int em = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  if ((unsigned)(em - 64) >= 0x7f8u - 64u) {
    if (!__any_sync(0xffffffffu, (b << 1) != 0)) return 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
  long long m = e ? ((b & 0xfffffffffffffLL) | (1LL << 52)) << 5 : 0;   // (subnormal: cut)
  m >>= min(em - e, 63);
  if (b < 0) m = -m;
  const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)m & 0x3ffffffu);
  const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(m >> 26) & 0x3ffffffu);
  const int s2 = __reduce_add_sync(0xffffffffu, (int)(m >> 52));
  const long long s = (long long)s0 + ((long long)s1 << 26) + ((long long)s2 << 52);
  if (s == 0) return 0.0;
  // |s| = u 2^-z with bit 63 of u set; the leading 53 bits, rounded, and the exponent
  unsigned long long u = s < 0 ? -(unsigned long long)s : (unsigned long long)s;
  const int z = __clzll((long long)u);
  u <<= z;
  const int ex = em + 6 - z;   // > 0: z <= 63
  const long long mag = ((long long)(ex - 1) << 52) + (long long)((u >> 11) + (u >> 10 & 1));
  return __longlong_as_double(mag | (s & (1LL << 63)));
}
// 1/x.  For 2^-1000 <= |x| < 2^1000: the reciprocal of the leading mantissa bits in FP32
// (relative error < 2^-21) with the exponent put in by integer instructions, then one cubic
// step r <- r + r (e + e^2), e = 1 - x r, which leaves e^3 < 2^-63: three FP64 operations.
// Comparing and converting in FP64 and two Newton-Raphson steps took eight.  Other x: IEEE
// division.
__device__ __forceinline__ double recip(double x) {
  const long long b = __double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  if ((unsigned)(e - 23) >= 2000u) return 1.0 / x;
  float f;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__int_as_float(0x3f800000 | ((int)(b >> 29) & 0x7fffff))));
  const double r = __longlong_as_double(((long long)__float_as_int(f) << 29) + ((long long)(896 + 1023 - e) << 52) |
                                        (b & (1LL << 63)));
  const double q = fma(-x, r, 1.0);
  return fma(r, fma(q, q, q), r);
}

// 1/sqrt(x) for 2^-1000 <= x < 2^1000: FP32 seed of the mantissa in [1, 4) with an even
// exponent, then one cubic step r <- r + r (e/2 + 3 e^2/8), e = 1 - x r^2.  Other x: IEEE sqrt.
__device__ __forceinline__ double rsqrt_pos(double x) {
  const long long b = __double_as_longlong(x);
  const int e = (int)(b >> 52);   // sign included
  if ((unsigned)(e - 23) >= 2000u) return 1.0 / sqrt(x);
  const int odd = (e & 1) ^ 1;    // biased by 1023: an even e is an odd exponent
  float f;
  asm("rsqrt.approx.ftz.f32 %0, %1;"
      : "=f"(f)
      : "f"(__int_as_float((0x3f800000 + (odd << 23)) | ((int)(b >> 29) & 0x7fffff))));
  const double r = __longlong_as_double(((long long)__float_as_int(f) << 29) +
                                        ((long long)(896 - ((e - 1023 - odd) >> 1)) << 52));
  const double t = x * r, q = fma(-t, r, 1.0);
  return fma(r * q, fma(q, 0.375, 0.5), r);
}

}  // namespace kscf
