// Degree step of the Chebyshev filter and Hamiltonian apply for FP64 blocks on 8^3 bricks
// (CheFSI paragraph of arXiv 2303.00790), slot-major rows:
//   out = alpha (H in - c in) + beta prev,
//   H in = -1/2 Lap_h in + V in + sum_i chi_i (E_i h^3 <chi_i, in>),
// the projections coming from kb_gather_kernel.
//
// The GB300 issues one FP64 warp instruction per 64 cycles and SM sub-partition, so the star is
// evaluated in integers (fixlap.cuh's weights): a CTA takes one brick and four vectors,
// converts the brick and its six halos once into 60-bit fixed point (in units of 2^-60 of 2^E, the
// power of two above the largest value of the vector in the brick and its neighbours, whose exponents
// every step writes for the next one, emax), and then every thread evaluates the 37-point sums of eight
// points from shared memory: 36 loads at register + constant addresses, five 64-bit additions per
// distance, fourteen 32 x 32 -> 64 products.  The sums are exact; FP64 is left for their
// conversion, the potential, the recurrence and the nonlocal term.
//
// Accuracy: no point's star is less accurate than in FP64, also where its neighbourhood lies far below
// 2^E.  A point whose own and next values are below S_STEEP gets its star apart (steep_points): the FP64
// star when a CTA has few of them, else from a second pass in a window 29 bits lower (a sum modulo
// 2^60, which the first pass's leading bits complete), and the FP64 star below 2^-36 of 2^E.  Measured
// against quadruple precision, error / (2^-53 sum |w v|) over fields exp(-r/2) .. exp(-4 r),
// Gaussians, waves and noise: rms 0.06-0.77 (FP64 star 0.22-0.94), largest 0.9-5.4 (0.9-5.4); filters of 8 to
// 12 steps with the recurrence's scalars as given: 1.3e-16 of a column's norm (FP64 star, whose
// seven weights are rounded, 6.0e-16 to 8.8e-16; the scalars' own rounding moves a result by 1e-15).
//
// What bounds it: the FP64 pipe (10.5 instructions per point and vector, 4.5 of them the nonlocal term
// with its divergence) is busy 40 % of the time, the rest is the load and conversion phase of 5.5
// values per point that two CTAs per SM hide half.  One degree step of 234,489 points x 850 vectors:
// 8.4 ms (gather 1.1 ms beside it) against 23.5 ms of the FP64 star; whole 12-step filter 295 -> 114 ms.
// Two limbs of 29 bits and no second look at small values took 102 ms, 105 ms 60 bits alone; a value of 1e-3
// of 2^E then had 47 bits, orbitals exp(-r) lost three digits in their tails.  What the small values'
// stars cost depends on the block: the orbitals of a self-consistent run, whose tails fill the shell
// outside the cluster, take 145 ms (with 64 or 512 for S_FEW 153 and 143); 200 orbitals exp(-r/2), exp(-r)
// or exp(-2 r) about as many centres, where most CTAs make the second pass, 40, 59 and 63 ms, FP64 star 70.
// Also built: the small values' stars one by one by the warp that meets them (120 to 137 ms: code that few
// warps run is fetched when it runs, and it shared the hot loop's registers), the 13-point sums as three
// line passes over register windows as in the FP32 filter, and 512 threads with half the planes each.
// A vector with a NaN, an Inf or nothing above 2^-767 in the brick or its neighbours takes the
// FP64 star, as do 16^3 bricks (cheb_step_generic).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fixlap.cuh"
#include "gather.cuh"
#include "kscf_internal.h"

namespace kscf {

namespace {

constexpr int S_BITS = 60;                       // |value| < 2^E -> |fixed| <= 2^60, unit 2^(E - 60)
constexpr int S_MULT = 56;                       // largest multiple of the integer weights, and twice the smallest
// Low bits of the sum that its conversion leaves out: the largest sum (21.2 2^E, 2^89.9 units) keeps 63 bits
constexpr int S_DROP = 27;
constexpr int S_FINE = 29;                       // the second window lies this many bits lower
// 5 |v| at the point + |v| at its six neighbours, 1/1.7 of what these put into sum |w v|, below
// which the sum is too coarse: 2^-6 of 2^E, in upper words (2^28 for 2^E).  The sum is off by at most
// 13.5 2^-60 2^E (cut values 10.6, S_DROP 2.9), so by 4 2^-53 sum |w v| at this line, where the FP64 star has
// 39 roundings; measured there 1.2 to 1.9, FP64 1.5 to 3.9.  (Twice the line: 0.4 to 1.6, 3 ms slower.)
constexpr uint32_t S_STEEP = 1u << 22;
constexpr int S_FEW = 192;                       // points of a CTA up to which they are taken one by one
constexpr int S_NV = 4;                          // vectors per CTA
constexpr int S_ENT = 256;                       // KB entries staged in shared memory
constexpr int S_THR = 256;                       // threads: 64 points of a plane x S_NV
// Shared memory: the fixed-point values of the brick and its halos, in points of S_NV x 8 bytes.
// Plane z = 0..7 of 256 points: the brick's 64 (x + 8 y), then the six points below and above
// every x line (6 y + q) and y line (8 q + x); behind the planes the 6 + 6 planes of the z halos.
constexpr int P_XL = 64, P_XH = 112, P_YL = 160, P_YH = 208, P_PLANE = 256, P_ZL = 8 * P_PLANE, P_ZH = P_ZL + 6 * 64,
              P_ALL = P_ZH + 6 * 64;
constexpr int S_FIX = 0, S_V = S_FIX + P_ALL * S_NV * 8, S_KBC = S_V + 512 * 8,
              S_CHI = S_KBC + KSCF_BRICK_ATOMS * 4 * S_NV * 8, S_EW = S_CHI + S_ENT * 32, S_KBP = S_EW + S_ENT * 4,
              S_LEFT = S_KBP + 514 * 2, S_SMEM = S_LEFT + 4 + S_FEW * 2;

// element (chunk c of S_NV columns, slot s, v) of a block at p[c * cs + s * ld + v]
struct Step64 {
  const double* in;
  int64_t cs_in, ld_in;
  const double* prev;   // may alias out (each element read before it is written)
  int64_t cs_prev, ld_prev;
  double* out;
  int64_t cs_out, ld_out;
  int n_cells, super;   // CTA order: supertiles of `super` bricks, chunk-major inside
  int w, nchunk, wq;    // columns, chunks of S_NV, row length of emax
  double alpha, beta, c;
  int wt[7];            // integer weights: m 831600 (3 w_0, w_1 .. w_6)
  uint32_t wabs[7];     // their magnitudes
  double ku;            // -1 / (2 h^2 831600 m)
  const double* coef;
  int64_t cld;
  const double* V;
  const int32_t* nbr;
  const uint8_t* mask;
  const int64_t* kb_ptr;
  const int32_t* kb_atom;
  const double* kb_chi;
  const uint32_t* eword;
  const int32_t *batoms, *bnat;
  const int *emax_in;
  int* emax_out;
  unsigned int* flag;   // with it, padding rows of out are zeroed and NaN or Inf in domain rows reported
  double st[7];
};

__device__ __forceinline__ uint32_t abs_hw(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }
// biased exponent of a maximum's high word; 0 only for zero
__device__ __forceinline__ int hw_exp(uint32_t hw) { return max((int)(hw >> 20), hw ? 1 : 0); }

// value -> floor(value 2^(S_BITS - E)) (negative values: one's complement).  What is cut off has
// the same mean everywhere and drops out of the star: its weights add up to zero.  e: the biased
// exponent with E = e - 1022.
__device__ __forceinline__ long long fix60(double v, int e) {
  const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
  const int n = min(e - (int)((h >> 20) & 0x7ff), 63);
  const uint32_t mh = (h & 0xfffffu) | 0x100000u;
  const unsigned long long t = ((((unsigned long long)mh << 32) | l) << (S_BITS - 53)) >> n;
  return (long long)(t ^ (unsigned long long)((long long)(int)h >> 31));
}
// the magnitude of a fixed-point value's upper word
__device__ __forceinline__ uint32_t abs_up(long long x) { return (uint32_t)abs((int)(x >> 32)); }
// the FP64 star at slot s of one column (bricks with non-finite or tiny values)
__device__ __noinline__ double star64(const Step64& a, const double* in, int64_t ld, int64_t s) {
  const int64_t brick = s >> 9;
  const int li = (int)(s & 511);
  const int l[3] = {li & 7, (li >> 3) & 7, li >> 6};
  const int stride[3] = {1, 8, 64};
  double acc = 3.0 * a.st[0] * in[s * ld];
  for (int ax = 0; ax < 3; ax++)
    for (int k = 1; k <= 6; k++) {
      double pair = 0.0;
      for (int sg = -1; sg <= 1; sg += 2) {
        const int n = l[ax] + sg * k;
        int64_t ns = s + (int64_t)sg * k * stride[ax];
        if (n < 0 || n >= 8) {
          const int nb = a.nbr[brick * 6 + 2 * ax + (sg > 0 ? 1 : 0)];
          if (nb < 0) continue;
          ns = (int64_t)nb * 512 + li + (sg * k - sg * 8) * stride[ax];
        }
        pair += in[ns * ld];
      }
      acc += a.st[k] * pair;
    }
  return acc;
}

// the same window of 60 bits, S_FINE bits lower: modulo 2^60
__device__ __forceinline__ long long fix60_low(double v, int e) {
  const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
  const int n = e - (int)((h >> 20) & 0x7ff) - S_FINE;
  const unsigned long long m = (((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32) | l) << (S_BITS - 53);
  const unsigned long long t = (n < 0 ? m << -n : m >> min(n, 63)) ^ (unsigned long long)((long long)(int)h >> 31);
  return (long long)(t << (64 - S_BITS)) >> (64 - S_BITS);
}
// a sum in units of 2^(E - S_BITS - S_FINE), |sum| < 2^119: its leading 63 bits; ku: the value
// of a unit of 2^(E - S_BITS)
__device__ __forceinline__ double sum_value(__int128 sum, double ku) {
  if (sum == 0) return 0.0;
  const unsigned __int128 m = sum < 0 ? -(unsigned __int128)sum : (unsigned __int128)sum;
  const unsigned long long mh = (unsigned long long)(m >> 64);
  const int z = mh ? __clzll((long long)mh) : 64 + __clzll((long long)(unsigned long long)m);
  const double r = (double)(long long)((unsigned long long)((m << z) >> 64) >> 1);   // in [2^62, 2^63]
  const double scale = __longlong_as_double(__double_as_longlong(ku) + ((long long)(65 - z - S_FINE) << 52));
  return sum < 0 ? -(r * scale) : r * scale;
}

// The FP64 star by eight lanes, one for each arm and one for the point itself; all lanes of the
// warp call it
__device__ __forceinline__ double star64_lanes(const Step64& a, const double* in, int64_t ld, int64_t s) {
  const int f = threadIdx.x & 7;
  double t = 0.0;
  if (f < 6) {
    const int li = (int)(s & 511), sh = 3 * (f >> 1), l = (li >> sh) & 7, room = (f & 1) ? 7 - l : l;
    const int st = (f & 1) ? 1 << sh : -(1 << sh), nb = __ldg(a.nbr + (s >> 9) * 6 + f);
    const int64_t out = (int64_t)nb * 512 + li - 8 * st;
    double v[6];
#pragma unroll
    for (int k = 1; k <= 6; k++)
      v[k - 1] = k <= room ? __ldg(in + (s + k * st) * ld) : nb >= 0 ? __ldg(in + (out + k * st) * ld) : 0.0;
#pragma unroll
    for (int k = 6; k >= 1; k--) t = fma(a.st[k], v[k - 1], t);
  } else if (f == 6) {
    t = 3.0 * a.st[0] * __ldg(in + s * ld);
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// the star's constant times 2^(e - 1022 - S_BITS)
__device__ __forceinline__ double unit_value(const Step64& a, int e) {
  return a.ku * __hiloint2double((e - 1022 - S_BITS + 1023) << 20, 0);
}

// The thread's vector of the brick from slot b0 and of its halos to fixed point: N rows 64 rows
// apart from row r0, to N points dstep apart
template <typename F>
__device__ __forceinline__ void stage_brick(long long* fx, const double* inc, int64_t ld, int64_t b0, const int (&nb)[6],
                                            bool on, int e, F fix) {
  const int v = threadIdx.x & 3, p = threadIdx.x >> 2, px = p & 7, py = p >> 3;
  auto stage = [&](auto n_c, bool use, int64_t r0, int dst, int dstep) {
    constexpr int N = decltype(n_c)::value;
    const double* src = inc + r0 * ld;
    double h[N];
#pragma unroll
    for (int q = 0; q < N; q++) h[q] = use ? __ldg(src + q * 64 * ld) : 0.0;
#pragma unroll
    for (int q = 0; q < N; q++) fx[(dst + q * dstep) * S_NV + v] = fix(h[q], e);
  };
  using I8 = std::integral_constant<int, 8>;
  using I6 = std::integral_constant<int, 6>;
  stage(I8(), on, b0 + p, p, P_PLANE);
  // x halos: px < 6 of every line; y halos: rows py < 6; planes z = 0..7
  if (px < 6) {
    stage(I8(), on && nb[0] >= 0, (int64_t)nb[0] * 512 + py * 8 + 2 + px, P_XL + py * 6 + px, P_PLANE);
    stage(I8(), on && nb[1] >= 0, (int64_t)nb[1] * 512 + p, P_XH + py * 6 + px, P_PLANE);
  }
  if (py < 6) {
    stage(I8(), on && nb[2] >= 0, (int64_t)nb[2] * 512 + (2 + py) * 8 + px, P_YL + p, P_PLANE);
    stage(I8(), on && nb[3] >= 0, (int64_t)nb[3] * 512 + p, P_YH + p, P_PLANE);
  }
  stage(I6(), on && nb[4] >= 0, (int64_t)nb[4] * 512 + 128 + p, P_ZL + p, 64);
  stage(I6(), on && nb[5] >= 0, (int64_t)nb[5] * 512 + p, P_ZH + p, 64);
}

// Byte offsets of the thread's point of plane 0 and of its neighbours along x and y (plane z is
// P_PLANE points further)
struct Arms {
  uint32_t me, x[12], y[12];
};
__device__ __forceinline__ Arms arms() {
  const int v = threadIdx.x & 3, p = threadIdx.x >> 2, px = p & 7, py = p >> 3;
  auto off = [&](int pt) { return (uint32_t)(pt * S_NV + v) * 8u; };
  Arms n;
  n.me = off(p);
#pragma unroll
  for (int k = 1; k <= 6; k++) {
    n.x[2 * k - 2] = off(px >= k ? p - k : P_XL + py * 6 + px - k + 6);
    n.x[2 * k - 1] = off(px + k < 8 ? p + k : P_XH + py * 6 + px + k - 8);
    n.y[2 * k - 2] = off(py >= k ? p - 8 * k : P_YL + (py - k + 6) * 8 + px);
    n.y[2 * k - 1] = off(py + k < 8 ? p + 8 * k : P_YH + (py + k - 8) * 8 + px);
  }
  return n;
}
// The star at the thread's point of plane z: hi 2^32 + lo, from the upper words with the signed
// weights and the lower words with their magnitudes in a positive (k odd) and a negative sum, one
// 32 x 32 -> 64 product each.  Returns what stands at the point and next to it (S_STEEP).
__device__ __forceinline__ uint32_t star60(const Step64& a, const long long* fx, const Arms& n, int z, long long& hi,
                                           long long& lo) {
  auto at = [&](uint32_t o, int imm) { return *(const long long*)((const char*)fx + o + imm); };
  constexpr int PL = P_PLANE * S_NV * 8;   // bytes of a plane
  auto zoff = [](int zz) {                 // plane zz, possibly in the z halos
    return zz < 0 ? (P_ZL + (zz + 6) * 64) * S_NV * 8 : zz > 7 ? (P_ZH + (zz - 8) * 64) * S_NV * 8 : zz * PL;
  };
  const long long x0 = at(n.me, z * PL);
  hi = (long long)a.wt[0] * (int)(x0 >> 32);
  unsigned long long neg = (unsigned long long)a.wabs[0] * (uint32_t)x0, pos = 0;
  uint32_t size = 0;
#pragma unroll
  for (int k = 1; k <= 6; k++) {
    const long long xa = at(n.x[2 * k - 2], z * PL), xb = at(n.x[2 * k - 1], z * PL), ya = at(n.y[2 * k - 2], z * PL),
                    yb = at(n.y[2 * k - 1], z * PL), za = at(n.me, zoff(z - k)), zb = at(n.me, zoff(z + k));
    const long long x = (xa + xb + ya) + (yb + za + zb);
    hi += (long long)a.wt[k] * (int)(x >> 32);
    if (k & 1) pos += (unsigned long long)a.wabs[k] * (uint32_t)x;
    else neg += (unsigned long long)a.wabs[k] * (uint32_t)x;
    if (k == 1)
      size = 5u * abs_up(x0) + (abs_up(xa) + abs_up(xb) + abs_up(ya)) + (abs_up(yb) + abs_up(za) + abs_up(zb));
  }
  lo = (long long)(pos - neg);
  return size;
}
// the sum in units of 2^S_DROP, rounded
__device__ __forceinline__ long long leading(long long hi, long long lo) {
  return (hi << (32 - S_DROP)) + ((lo + (1ll << (S_DROP - 1))) >> S_DROP);
}

// Adds alpha times the star where the first pass left it out (`left`: planes of the thread's
// point).  Called by all threads; apart from the kernel, whose registers it does not share.
//   Few points: the FP64 star, four points a warp at a time.
//   More: the whole brick once more in the window S_FINE bits lower, which gives the sum modulo
// 2^60; the leading bits of the first pass, off by less than 2^58.2, give the rest.  Where that is
// too coarse as well, the FP64 star.
template <bool CM>
__device__ __noinline__ void steep_points(const Step64& a, uint8_t* smb, int cell, int chunk, int e, uint32_t left,
                                          int* s_max) {
  long long* fx = (long long*)(smb + S_FIX);
  int* count = (int*)(smb + S_LEFT);
  uint16_t* list = (uint16_t*)(count + 1);   // point * S_NV + vector
  const int64_t ld = CM ? S_NV : a.ld_in, b0 = (int64_t)cell * 512;
  const int tid = threadIdx.x, v = tid & 3, p = tid >> 2;
  const double* in = a.in + (int64_t)chunk * a.cs_in;
  auto add = [&](int r, int vec, double t) {
    double* o = a.out + (int64_t)chunk * a.cs_out + vec + (b0 + r) * a.ld_out;
    t = fma(a.alpha, t, *o);
    *o = t;
    if (a.flag && abs_hw(t) >= 0x7ff00000u) atomicOr(a.flag, 1u);
    if (a.emax_out) atomicMax(&s_max[vec], hw_exp(abs_hw(t)));
  };
#pragma unroll 1
  for (uint32_t m = left; m; m &= m - 1) {
    const int i = atomicAdd(count, 1);
    if (i < S_FEW) list[i] = (uint16_t)(((__ffs(m) - 1) * 64 + p) * S_NV + v);
  }
  __syncthreads();
  const int n = *count;
  if (n <= S_FEW) {
    for (int i0 = tid / 32 * 4; i0 < n; i0 += S_THR / 8) {
      const int i = i0 + (tid & 31) / 8, item = list[min(i, n - 1)], vec = item & (S_NV - 1), r = item / S_NV;
      const double t = star64_lanes(a, in + vec, ld, b0 + r);
      if ((tid & 7) == 0 && i < n) add(r, vec, t);
    }
    return;
  }
  const Arms at = arms();
  long long lead[8], hi, lo;
#pragma unroll 1
  for (uint32_t m = left; m; m &= m - 1) {
    const int z = __ffs(m) - 1;
    star60(a, fx, at, z, hi, lo);
    lead[z] = leading(hi, lo);
  }
  __syncthreads();
  int nb[6];
#pragma unroll
  for (int f = 0; f < 6; f++) nb[f] = __ldg(a.nbr + (int64_t)cell * 6 + f);
  stage_brick(fx, in + v, ld, b0, nb, chunk * S_NV + v < a.w, e, [](double h, int ex) { return fix60_low(h, ex); });
  __syncthreads();
#pragma unroll 1
  for (; left; left &= left - 1) {
    const int z = __ffs(left) - 1;
    double t;
    if (star60(a, fx, at, z, hi, lo) < S_STEEP) {
      t = star64(a, in + v, ld, b0 + z * 64 + p);
    } else {
      const __int128 low = ((__int128)hi << 32) + lo, rest = ((__int128)lead[z] << (S_DROP + S_FINE)) - low;
      t = sum_value(low + ((rest + ((__int128)1 << (S_BITS - 1))) >> S_BITS << S_BITS), unit_value(a, e));
    }
    add(z * 64 + p, v, t);
  }
}

// SMEM_KB: the bricks have at most KSCF_BRICK_ATOMS atoms with projectors (so that 16 bits hold
// the number of an entry inside its brick), whose coefficients are staged in shared memory with
// the first S_ENT entries
static_assert(KSCF_BRICK_ATOMS * 512 < 65536, "entry numbers of a brick in 16 bits");
// CM: `in` is chunk-major (ld_in = S_NV)
template <bool SMEM_KB, bool CM>
__global__ void __launch_bounds__(S_THR, 2) step64_kernel(const __grid_constant__ Step64 a) {
  extern __shared__ __align__(16) uint8_t smb[];
  long long* fx = (long long*)(smb + S_FIX);   // [point][4]
  double* vs = (double*)(smb + S_V);           // [512]: V
  double* kbc = (double*)(smb + S_KBC);        // [atom][l][4]
  double* echi = (double*)(smb + S_CHI);       // [entry][4]
  uint32_t* ew = (uint32_t*)(smb + S_EW);
  uint16_t* kbp = (uint16_t*)(smb + S_KBP);    // [513]: first entry of each point (SMEM_KB)
  __shared__ int s_max[S_NV];
  int cell, chunk;
  {
    const int per = a.nchunk * a.super, t = blockIdx.x / per, rem = blockIdx.x - t * per;
    chunk = rem / a.super;
    cell = t * a.super + rem - chunk * a.super;
    if (cell >= a.n_cells) return;
  }
  const int64_t ld = CM ? S_NV : a.ld_in;
  const int tid = threadIdx.x, v = tid & 3, p = tid >> 2;   // p: the thread's point of every plane
  const int col = chunk * S_NV + v;
  const bool on = col < a.w;
  const int64_t b0 = (int64_t)cell * 512;
  if (tid < S_NV) s_max[tid] = 0;
  if (tid == 0) *(int*)(smb + S_LEFT) = 0;
  int nb[6];
#pragma unroll
  for (int f = 0; f < 6; f++) nb[f] = __ldg(a.nbr + (int64_t)cell * 6 + f);
  const double* inc = a.in + (int64_t)chunk * a.cs_in + v;
  // exponent of the vector over the brick and its neighbours
  int e = 0;
  if (on) {
    e = __ldg(a.emax_in + (int64_t)cell * a.wq + col);
#pragma unroll
    for (int f = 0; f < 6; f++)
      if (nb[f] >= 0) e = max(e, __ldg(a.emax_in + (int64_t)nb[f] * a.wq + col));
  }
  const int64_t e0 = __ldg(a.kb_ptr + b0), e1 = __ldg(a.kb_ptr + b0 + 512);
  for (int t = tid; t < 512; t += S_THR) vs[t] = __ldg(a.V + b0 + t);
  if (SMEM_KB) {
    for (int t = tid; t <= 512; t += S_THR) kbp[t] = (uint16_t)(__ldg(a.kb_ptr + b0 + t) - e0);
    const int nat = __ldg(a.bnat + cell);
    for (int t = tid; t < nat * 4 * S_NV; t += S_THR) {
      const int at = __ldg(a.batoms + (int64_t)cell * KSCF_BRICK_ATOMS + t / (4 * S_NV)), l = (t / S_NV) & 3;
      const int cc = chunk * S_NV + (t & (S_NV - 1));
      kbc[t] = cc < a.w ? a.coef[((int64_t)at * 4 + l) * a.cld + cc] : 0.0;
    }
    const int ne = (int)min(e1 - e0, (int64_t)S_ENT);
    for (int t = tid; t < ne; t += S_THR) {
      ew[t] = __ldg(a.eword + e0 + t);
      *(double2*)(echi + 4 * t) = __ldg((const double2*)(a.kb_chi + 4 * (e0 + t)));
      *(double2*)(echi + 4 * t + 2) = __ldg((const double2*)(a.kb_chi + 4 * (e0 + t)) + 1);
    }
  }
  // a vector of zeros (some may be -0, one unit below): its star is zero
  const bool zero = e == 0;
  // the value of a unit of the sum (used when not slow); the FP64 star also where it is not well
  // inside the normal numbers
  const double ku = unit_value(a, e);
  const bool slow = __syncthreads_or(!zero && (e >= 2046 || e < 256 || (int)(abs_hw(ku) >> 20) < 200));
  if (zero) e = 1023;
  const double ku_d = zero ? 0.0 : ku * (double)(1 << S_DROP);
  if (!slow) stage_brick(fx, inc, ld, b0, nb, on, e, [](double h, int ex) { return fix60(h, ex); });
  // ---- the point's own value, prev and mask of all planes, before the first store (plain loads
  // of prev: it may be the output) ----
  double yv[8], pv[8];
  uint32_t live = 0;
  {
    const double* prevc = a.prev + (int64_t)chunk * a.cs_prev + v + (b0 + p) * a.ld_prev;
#pragma unroll
    for (int z = 0; z < 8; z++) live |= (uint32_t)(__ldg(a.mask + b0 + z * 64 + p) != 0) << z;
    if (!on) live = 0;
#pragma unroll
    for (int z = 0; z < 8; z++) {
      const bool use = (live >> z) & 1u;
      yv[z] = use ? __ldg(inc + (b0 + z * 64 + p) * ld) : 0.0;
      pv[z] = use && a.prev ? prevc[z * 64 * a.ld_prev] : 0.0;
    }
  }
  const Arms at = arms();
  __syncthreads();   // the fixed-point values, V and the KB tables are visible
  uint32_t mx = 0, left = 0;   // left: planes of points that steep_points adds the star to
  double* outc = a.out + (int64_t)chunk * a.cs_out + v + (b0 + p) * a.ld_out;
  const uint32_t limit = zero ? 0u : S_STEEP;
#pragma unroll
  for (int z = 0; z < 8; z++) {
    if (!((live >> z) & 1u)) {
      if (a.flag && on) outc[z * 64 * a.ld_out] = 0.0;
      continue;
    }
    const int r = z * 64 + p;
    double t;
    bool steep = false;
    if (slow) {
      t = star64(a, inc, ld, b0 + r);
    } else {
      long long hi, lo;
      steep = star60(a, fx, at, z, hi, lo) < limit;
      t = ku_d * (double)leading(hi, lo);
      if (steep) {   // without its star for now
        t = 0.0;
        left |= 1u << z;
      }
    }
    t = fma(vs[r], yv[z], t);
    if (SMEM_KB) {
      for (int i = kbp[r], i1 = kbp[r + 1]; i < i1; i++) {
        const int64_t qe = e0 + i;
        uint32_t word;
        double2 c0, c1;
        if (i < S_ENT) {
          word = ew[i];
          c0 = *(const double2*)(echi + 4 * i);
          c1 = *(const double2*)(echi + 4 * i + 2);
        } else {
          word = __ldg(a.eword + qe);
          c0 = __ldg((const double2*)(a.kb_chi + 4 * qe));
          c1 = __ldg((const double2*)(a.kb_chi + 4 * qe) + 1);
        }
        const double* cf = kbc + (word >> 16) * (4 * S_NV) + v;
        t = fma(c0.x, cf[0], t);
        t = fma(c0.y, cf[S_NV], t);
        t = fma(c1.x, cf[2 * S_NV], t);
        t = fma(c1.y, cf[3 * S_NV], t);
      }
    } else {   // any number of entries in the brick
      for (int64_t qe = __ldg(a.kb_ptr + b0 + r), q1 = __ldg(a.kb_ptr + b0 + r + 1); qe < q1; qe++) {
        const double* cf = a.coef + (int64_t)__ldg(a.kb_atom + qe) * 4 * a.cld + col;
        const double* ch = a.kb_chi + 4 * qe;
        t = fma(ch[0], cf[0], t);
        t = fma(ch[1], cf[a.cld], t);
        t = fma(ch[2], cf[2 * a.cld], t);
        t = fma(ch[3], cf[3 * a.cld], t);
      }
    }
    t = fma(a.beta, pv[z], a.alpha * fma(-a.c, yv[z], t));
    outc[z * 64 * a.ld_out] = t;
    mx = max(mx, steep ? 0u : abs_hw(t));
  }
  if (__syncthreads_or(left != 0)) steep_points<CM>(a, smb, cell, chunk, e, left, s_max);
  if (a.flag && mx >= 0x7ff00000u) atomicOr(a.flag, 1u);
  if (a.emax_out) {
    // lanes of the same vector are 4 apart
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) < S_NV) atomicMax(&s_max[v], hw_exp(mx));
    __syncthreads();
    if (tid < S_NV && chunk * S_NV + tid < a.w) a.emax_out[(int64_t)cell * a.wq + chunk * S_NV + tid] = s_max[tid];
  }
}

// emax[brick][v] = exponent of max |X| over the brick's domain rows: one CTA per brick and 32
// columns
__global__ void __launch_bounds__(256) emax_kernel(const double* __restrict__ X, int64_t ld, int w, int wq,
                                                   const uint8_t* __restrict__ mask, int* __restrict__ emax) {
  __shared__ uint32_t red[8][32];
  const int col = blockIdx.y * 32 + (threadIdx.x & 31), wy = threadIdx.x >> 5;
  const int64_t b0 = (int64_t)blockIdx.x * 512;
  uint32_t m = 0;
  if (col < w) {
#pragma unroll 4
    for (int r = wy; r < 512; r += 8)
      if (__ldg(mask + b0 + r)) m = max(m, (uint32_t)__double2hiint(__ldg(X + (b0 + r) * ld + col)) & 0x7fffffffu);
  }
  red[wy][threadIdx.x & 31] = m;
  __syncthreads();
  if (wy == 0 && col < w) {
#pragma unroll
    for (int q = 1; q < 8; q++) m = max(m, red[q][threadIdx.x]);
    emax[(int64_t)blockIdx.x * wq + col] = hw_exp(m);
  }
}

// Chunk-major copy A of w columns of a slot-major block (padded columns and padding rows zero,
// padding rows not read), the padding rows of the second working copy B zeroed too, and the
// exponents of the bricks: one CTA per brick and 32 columns.
__global__ void __launch_bounds__(256) to_cm64_kernel(const double* __restrict__ X, int64_t ld, int w, int wq,
                                                      int64_t n_slots, const uint8_t* __restrict__ mask,
                                                      double* __restrict__ A, double* __restrict__ B,
                                                      int* __restrict__ emax) {
  __shared__ uint32_t red[8][32];
  const int lane = threadIdx.x & 31, col = blockIdx.y * 32 + lane, wy = threadIdx.x >> 5;
  const int64_t b0 = (int64_t)blockIdx.x * 512, o = (int64_t)(col / S_NV) * n_slots * S_NV + (col & (S_NV - 1));
  uint32_t m = 0;
  if (col < wq) {
#pragma unroll 4
    for (int r = wy; r < 512; r += 8) {
      const int64_t s = b0 + r;
      const bool live = __ldg(mask + s) != 0;
      const double x = live && col < w ? __ldg(X + s * ld + col) : 0.0;
      A[o + s * S_NV] = x;
      if (!live) B[o + s * S_NV] = 0.0;
      m = max(m, (uint32_t)__double2hiint(x) & 0x7fffffffu);
    }
  }
  red[wy][lane] = m;
  __syncthreads();
  if (wy == 0 && col < w) {
#pragma unroll
    for (int q = 1; q < 8; q++) m = max(m, red[q][lane]);
    emax[(int64_t)blockIdx.x * wq + col] = hw_exp(m);
  }
}

int emax_ld(int w) { return (w + 3) / 4 * 4; }

constexpr int kFixW[6] = {1425600, -222750, 44000, -7425, 864, -50};

// The star's one floating-point constant is -1 / (2 h^2 831600 m); its rounding error would be a
// systematic relative error of the kinetic energy in every step.  The weights may be taken any
// S_MULT/2 < m <= S_MULT times: the m whose constant is closest to a double (a smaller m has
// the error of twice its value).
int weight_multiple(double h, double* ku) {
  const double hh = h * h, hl = std::fma(h, h, -hh);   // h^2 = hh + hl exactly
  int best = S_MULT;
  double err = 1.0;
  for (int m = S_MULT / 2 + 1; m <= S_MULT; m++) {
    const double d = 2.0 * FIX_DEN * m, p = d * hh, pl = std::fma(d, hh, -p) + d * hl, u = 1.0 / p;
    const double q = u * p, r = std::fabs(((1.0 - q) - std::fma(u, p, -q)) - u * pl);   // |1 - u d h^2|
    if (r < err) {
      err = r;
      best = m;
      *ku = -u;
    }
  }
  return best;
}

}  // namespace

bool step64_available(const Ham& H) { return H.grid.B == 8 && H.n_cells == H.grid.n_bricks && H.n_cells > 0; }

// A single application also needs the exponents' pass: measured, us, this path | FP64 star:
// 4,169 points x 8 39 | 29, x 32 43 | 43, 8,925 x 16 40 | 44, 45,025 x 1 50 | 37, x 2 50 | 44, x 4 50 | 50 (three
// launches of 12 us and more each), 97,569 x 1 54 | 46
bool step64_wanted(const Ham& H, int w) { return step64_available(H) && (double)H.grid.n_points * w >= 1.5e5; }

// A filter's block goes through in `parts`, one after the other, each with a gather and a step per
// degree that a small grid does not fill.  Measured, us per degree: this path 31 for every part + 4e-5 for
// every value (points x columns), the FP64 star 25 + 1.1e-4.  Whole filters of 10 degrees, this path | FP64
// star: 4,169 points x 8 (1 part) 323 | 260, x 32 (3) 963 | 404, x 100 (2) 841 | 717; 8,925 x 8 (1) 327 | 324, x 48
// (2) 755 | 709; 17,557 x 8 (1) 329 | 419, x 24 (2) 730 | 723, x 36 (2) 815 | 961, x 32 (3) 1043 | 858, x 64 (3)
// 1299 | 1491; 33,401 x 1 (1) 344 | 302, x 28 (3) 1175 | 1317; 45,025 x 128 (3) 3453 | 7094
bool step64_filter_wanted(const Ham& H, int w, int parts) {
  return step64_available(H) && 30.0 * parts - 26.0 < 7.5e-5 * (double)H.grid.n_points * w;
}

size_t step64_emax_bytes(const Ham& H, int w) { return kscf_align256((size_t)H.grid.n_bricks * emax_ld(w) * 4); }

cudaError_t launch_emax64(const Ham& H, const double* X, int64_t ld, int w, int* emax, cudaStream_t st) {
  emax_kernel<<<dim3((unsigned)H.grid.n_bricks, (w + 31) / 32), 256, 0, st>>>(X, ld, w, emax_ld(w), H.d_mask, emax),
      count_launch();
  return cudaGetLastError();
}

cudaError_t launch_to_cm64(const Ham& H, const double* X, int64_t ld, int w, double* A, double* B, int* emax,
                           cudaStream_t st) {
  to_cm64_kernel<<<dim3((unsigned)H.grid.n_bricks, (w + 31) / 32), 256, 0, st>>>(X, ld, w, emax_ld(w), H.grid.n_slots,
                                                                                H.d_mask, A, B, emax),
      count_launch();
  return cudaGetLastError();
}

cudaError_t launch_gather_cm64(const Ham& H, const double* Y, int w, double* coef, int64_t cld, cudaStream_t st) {
  if (H.n_kb == 0 || w == 0) return cudaSuccess;
  count_launch();
  return launch_gather<double, 2>({Y, H.grid.n_slots * S_NV, S_NV, 2, w, 0, cld, H.d_kb_atom_ptr, H.d_kb_atom_slot,
                                   H.d_kb_atom_chi64, H.d_kb_energy, coef},
                                  H.n_kb, st);
}

// ld < 0: chunk-major
cudaError_t launch_step64(const Ham& H, const double* in, int64_t ld_in, const double* prev, int64_t ld_prev, double* out,
                          int64_t ld_out, int w, double alpha, double beta, double c, const double* coef, int64_t cld,
                          const int* emax_in, int* emax_out, cudaStream_t st, unsigned int* flag) {
  Step64 a;
  a.flag = flag;
  const bool cm = ld_in < 0;
  auto place = [&](int64_t ld, int64_t* cs, int64_t* l) {
    *cs = ld < 0 ? H.grid.n_slots * S_NV : S_NV;
    *l = ld < 0 ? S_NV : ld;
  };
  a.in = in;
  place(ld_in, &a.cs_in, &a.ld_in);
  a.prev = prev;
  place(ld_prev, &a.cs_prev, &a.ld_prev);
  a.out = out;
  place(ld_out, &a.cs_out, &a.ld_out);
  a.w = w;
  a.nchunk = (w + S_NV - 1) / S_NV;
  a.wq = emax_ld(w);
  a.n_cells = (int)H.grid.n_bricks;
  // chunk-major: the bricks of one chunk stay in L2 (three copies of 16 KB each); slot-major:
  // all chunks of a brick side by side, so that the sectors of its rows are used together
  a.super = cm ? (int)std::max<int64_t>(64, std::min<int64_t>(H.grid.n_bricks, (64LL << 20) / (3 * 512 * S_NV * 8))) : 1;
  a.alpha = alpha;
  a.beta = beta;
  a.c = c;
  const int m = weight_multiple(H.grid.h, &a.ku);
  a.wt[0] = m * FIX_W0;
  for (int k = 1; k <= 6; k++) a.wt[k] = m * kFixW[k - 1];
  for (int k = 0; k <= 6; k++) a.wabs[k] = (uint32_t)std::abs(a.wt[k]);
  a.coef = coef;
  a.cld = cld;
  a.V = H.d_v64;
  a.nbr = H.d_nbr;
  a.mask = H.d_mask;
  a.kb_ptr = H.d_kb_slot_ptr;
  a.kb_atom = H.d_kb_slot_atom;
  a.kb_chi = H.d_kb_slot_chi64;
  a.eword = H.d_kb_entry_word;
  a.batoms = H.d_brick_atoms;
  a.bnat = H.d_brick_natoms;
  a.emax_in = emax_in;
  a.emax_out = emax_out;
  for (int k = 0; k < 7; k++) a.st[k] = H.stencil[k];
  const int64_t n_super = (H.grid.n_bricks + a.super - 1) / a.super;
  const unsigned grid = (unsigned)(n_super * a.super * a.nchunk);
  auto run = [&](auto kern) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S_SMEM);
    if (e != cudaSuccess) return e;
    kern<<<grid, S_THR, S_SMEM, st>>>(a), count_launch();
    return cudaGetLastError();
  };
  if (H.brick_atoms_ok) return cm ? run(step64_kernel<true, true>) : run(step64_kernel<true, false>);
  return cm ? run(step64_kernel<false, true>) : run(step64_kernel<false, false>);
}

}  // namespace kscf
