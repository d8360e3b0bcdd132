// Fixed-point evaluation of the order-12 Laplacian for FP64 fields.
//
// The GB300 issues one FP64 warp instruction per 64 cycles and SM sub-partition, so the
// 37-term FP64 star costs ~2,400 cycles per 32 points.  Its weights are rationals with the
// common denominator 831600 (w_k = 2 (-1)^{k+1} (6!)^2 / (k^2 (6-k)! (6+k)!)), so with the
// field held as 58-bit fixed-point numbers the star is exact integer arithmetic on the
// full-rate pipes: per distance k the six neighbours are added in 32 bits per limb and
// multiplied by the integer weight into 64-bit sums.  What is rounded is the conversion of
// the field (to 2^-57 of its bound: 2^-53 of every value within 2^-4 of it) and the sum, once,
// when it becomes FP64; the FP64 star rounds after each of its 37 operations.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace kscf {

constexpr int FIX_BITS = 57;          // |value| < 2^E  ->  |fixed| <= 2^57
constexpr int FIX_LO = 29;            // fixed = hi * 2^29 + lo, -2^28 <= lo < 2^28, |hi| <= 2^28
constexpr double FIX_DEN = 831600.0;  // common denominator of the weights
// 831600 w_k, k = 1..6, and 831600 * 3 w_0; sum over the star of |weights| < 2^24.1
constexpr int FIX_W0 = -7441434;
__device__ constexpr int FIX_W[6] = {1425600, -222750, 44000, -7425, 864, -50};

// biased exponent e with |value| < 2^(e - 1022) for every |value| whose high word is at
// most hw (sign cleared)
__device__ __forceinline__ int fix_exp(uint32_t hw) { return (int)(hw >> 20); }

// value -> round(value 2^(FIX_BITS - (e - 1022))) as (hi, lo) limbs; integer instructions only
__device__ __forceinline__ int2 fix_from(double v, int e) {
  const long long b = __double_as_longlong(v);
  int ev = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (ev) m |= 1ull << 52;
  else ev = 1;
  const int sh = ev - e + (FIX_BITS - 53);
  unsigned long long t;
  if (sh >= 0) {
    t = m << min(sh, FIX_BITS - 52);
  } else {
    const int n = min(-sh, 60);
    t = (m + (1ull << (n - 1))) >> n;
  }
  const long long x = b < 0 ? -(long long)t : (long long)t;
  const int lo = (int)((uint32_t)x << (32 - FIX_LO)) >> (32 - FIX_LO);
  return make_int2((int)((x - lo) >> FIX_LO), lo);
}

// sums of one point: s.x = sum_k W_k (sum of hi limbs), s.y the same of the lo limbs
struct FixAcc {
  long long hi, lo;
};
__device__ __forceinline__ void fix_mad(FixAcc& a, int w, int2 s) {
  a.hi += (long long)w * s.x;
  a.lo += (long long)w * s.y;
}
__device__ __forceinline__ int2 fix_add(int2 a, int2 b) { return make_int2(a.x + b.x, a.y + b.y); }
// The sum in units of FIX_SUM_UNIT fixed-point units: hi 2^29 + lo without its last 19 bits
// (2^-62 of the largest sum the bound allows), rounded to FP64 by one conversion
constexpr double FIX_SUM_UNIT = 524288.0;   // 2^19
__device__ __forceinline__ double fix_value(const FixAcc& a) {
  return (double)((a.hi << (FIX_LO - 19)) + (a.lo >> 19));
}
// 2^(e - 1022 - FIX_BITS): one fixed-point unit
__device__ __forceinline__ double fix_unit(int e) {
  const int b = e - 1022 - FIX_BITS + 1023;   // its biased exponent
  return b >= 1 ? __hiloint2double(b << 20, 0) : scalbn(1.0, e - 1022 - FIX_BITS);
}

}  // namespace kscf
