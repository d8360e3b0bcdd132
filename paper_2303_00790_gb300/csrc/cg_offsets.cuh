// Byte offsets into the CG's fixed-point field (8 bytes a slot), from a base one brick of B^3 slots
// before the field, so that no offset is negative (that of a high neighbour starts below the neighbour's
// first slot).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define KSCF_HD __host__ __device__ __forceinline__
#else
#define KSCF_HD inline
#endif

namespace kscf {

// 32 bits keep the address arithmetic out of the loads (904,089 points: 23.0 ms a solve, 23.7 with
// 64).  They hold fields below 4 GB, 2^29 slots, with the base brick and the zeros behind; larger
// ones take 64.
KSCF_HD bool cg_wide(int64_t n, int zero_slots, int B) {
  return 8 * (n + zero_slots + 2 * B * B * B) > 0xffffffffll;
}

template <typename O, int B>
KSCF_HD O cg_own(int s) {
  return 8 * ((O)s + B * B * B);
}
// The zeros behind a field of n slots, zero_slots of them
template <typename O>
KSCF_HD O cg_zero(int64_t n, int zero_slots) {
  return 8 * (O)(n + zero_slots / 2);
}
// Face f = 2 axis + side of a slot that is number li of its brick, with neighbour brick n: +- 8 k stride
// from it is the slot at distance k beyond the face.  A missing brick (n < 0) points into the zeros.
template <typename O, int B>
KSCF_HD O cg_face(int n, int li, int f, O zero) {
  constexpr int B3 = B * B * B;
  const int ax = f >> 1, stride = ax == 0 ? 1 : ax == 1 ? B : B * B;
  return n >= 0 ? 8 * ((O)n * B3 + (O)(B3 + li + ((f & 1) ? -B : B) * stride)) : zero + 8 * B3;
}

}  // namespace kscf
