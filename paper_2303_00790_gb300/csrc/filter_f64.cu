// Degree step of the Chebyshev filter and Hamiltonian apply for FP64 blocks on 8^3 bricks
// (CheFSI paragraph of arXiv 2303.00790), slot-major rows:
//   out = alpha (H in - c in) + beta prev,
//   H in = -1/2 Lap_h in + V in + sum_i chi_i (E_i h^3 <chi_i, in>),
// the projections coming from kb_gather_kernel.
//
// The GB300 issues one FP64 warp instruction per 64 cycles and SM sub-partition, so the star is
// evaluated in integers (fixlap.cuh's weights): a CTA takes one brick and four vectors,
// converts the brick and its six halos once into 57-bit fixed point in two limbs (in units of
// the largest value of the vector in the brick and its neighbours, whose exponents every step
// writes for the next one, emax), and then every thread evaluates the 37-point sums of eight
// points from shared memory: 36 loads at register + constant addresses, six additions of 32
// bits per limb and distance, seven 32 x 32 -> 64 products per limb.  The sums are exact; FP64 is
// left for their conversion, the potential, the recurrence and the nonlocal term.
// What bounds it: the FP64 pipe is 43 % busy (10.5 instructions per point and vector, 4.5 of them
// the nonlocal term with its divergence), the rest is the load and conversion phase of 5.5 values per
// point that two CTAs per SM hide half.  One degree step of 234,489 points x 850 vectors: 7.4 ms
// (gather 1.1 ms beside it) against 23.5 ms of the FP64 star; whole 12-step filter 295 -> 101 ms.
// Also built: the 13-point sums as three line passes over register windows as in the FP32
// filter, three CTAs per SM (6.4 ms, but a less accurate order of the last operations), and 512
// threads with half the planes each (7.9 ms).  Error after 10 steps against extended precision:
// 1.6-2.4e-16 per column, FP64 star 2.4-3.3e-16.
// A vector with a NaN, an Inf or values below 2^-895 in the brick or its neighbours takes the
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

constexpr int S_BITS = 57;                       // |value| < 2^E -> |fixed| <= 2^57, unit 2^(E - 57)
constexpr int S_MULT = 64;                       // largest multiple of the integer weights
constexpr int S_DROP = 25;                       // low bits of the sum not kept (2^-62 of the largest sum)
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
              S_SMEM = S_KBP + 514 * 2;

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
  double ku;            // -2^S_DROP / (2 h^2 831600 m)
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

// value -> floor(value 2^(S_BITS - E)) (negative values: one's complement) as limbs hi 2^29 + lo,
// lo in [0, 2^29) stored less 2^28 so that six of them add up in 32 bits.  That constant, and the
// mean of what is cut off, drop out of the star: its weights add up to zero.  e: the biased
// exponent with E = e - 1022.
__device__ __forceinline__ int2 fix57(double v, int e) {
  const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
  const int n = min(e - (int)((h >> 20) & 0x7ff), 63);
  const uint32_t mh = (h & 0xfffffu) | 0x100000u;
  unsigned long long t = (((unsigned long long)mh << 32) | l) << (S_BITS - 53);
  t >>= n;
  const unsigned long long x = t ^ (unsigned long long)((long long)(int)h >> 31);
  return make_int2((int)(uint32_t)(x >> FIX_LO), (int)((uint32_t)x & ((1u << FIX_LO) - 1)) - (1 << (FIX_LO - 1)));
}

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

// SMEM_KB: the bricks have at most KSCF_BRICK_ATOMS atoms with projectors (so that 16 bits hold
// the number of an entry inside its brick), whose coefficients are staged in shared memory with
// the first S_ENT entries
static_assert(KSCF_BRICK_ATOMS * 512 < 65536, "entry numbers of a brick in 16 bits");
// CM: `in` is chunk-major (ld_in = S_NV)
template <bool SMEM_KB, bool CM>
__global__ void __launch_bounds__(S_THR, 2) step64_kernel(Step64 a) {
  extern __shared__ __align__(16) uint8_t smb[];
  int2* fx = (int2*)(smb + S_FIX);             // [point][4]
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
  const int px = p & 7, py = p >> 3;
  const int col = chunk * S_NV + v;
  const bool on = col < a.w;
  const int64_t b0 = (int64_t)cell * 512;
  if (tid < S_NV) s_max[tid] = 0;
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
  const bool slow = __syncthreads_or(e >= 2046 || (e > 0 && e < 128));
  // a vector of zeros (some may be -0, one unit below): its star is zero
  const double ku = e == 0 ? 0.0 : a.ku * fix_unit(e);
  if (e == 0) e = 1023;
  // ---- values to fixed point (S_BITS = FIX_BITS): N rows `step` rows apart from row r0, to N
  // points dstep apart ----
  if (!slow) {
    auto stage = [&](auto n_c, bool use, int64_t r0, int dst, int dstep) {
      constexpr int N = decltype(n_c)::value;
      const double* src = inc + r0 * ld;
      double h[N];
#pragma unroll
      for (int q = 0; q < N; q++) h[q] = use ? __ldg(src + q * 64 * ld) : 0.0;
#pragma unroll
      for (int q = 0; q < N; q++) fx[(dst + q * dstep) * S_NV + v] = fix57(h[q], e);
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
  // neighbour points of plane 0 along x and y (byte offsets; plane z is P_PLANE points further)
  uint32_t xo[12], yo[12];
  auto off = [&](int pt) { return (uint32_t)(pt * S_NV + v) * 8u; };
#pragma unroll
  for (int k = 1; k <= 6; k++) {
    xo[2 * k - 2] = off(px >= k ? p - k : P_XL + py * 6 + px - k + 6);
    xo[2 * k - 1] = off(px + k < 8 ? p + k : P_XH + py * 6 + px + k - 8);
    yo[2 * k - 2] = off(py >= k ? p - 8 * k : P_YL + (py - k + 6) * 8 + px);
    yo[2 * k - 1] = off(py + k < 8 ? p + 8 * k : P_YH + (py + k - 8) * 8 + px);
  }
  const uint32_t me = off(p);
  __syncthreads();   // the fixed-point values, V and the KB tables are visible
  uint32_t mx = 0;
  double* outc = a.out + (int64_t)chunk * a.cs_out + v + (b0 + p) * a.ld_out;
  const char* fb = (const char*)fx;
  constexpr int PL = P_PLANE * S_NV * 8;   // bytes of a plane
#pragma unroll
  for (int z = 0; z < 8; z++) {
    if (!((live >> z) & 1u)) {
      if (a.flag && on) outc[z * 64 * a.ld_out] = 0.0;
      continue;
    }
    const int r = z * 64 + p;
    double t;
    if (slow) {
      t = star64(a, inc, ld, b0 + r);
    } else {
      auto at = [&](uint32_t o, int imm) { return *(const int2*)(fb + o + imm); };
      // plane zz, possibly in the z halos (compile time)
      auto zoff = [](int zz) {
        return zz < 0 ? (P_ZL + (zz + 6) * 64) * S_NV * 8 : zz > 7 ? (P_ZH + (zz - 8) * 64) * S_NV * 8 : zz * PL;
      };
      FixAcc s = {0, 0};
      fix_mad(s, a.wt[0], at(me, z * PL));
#pragma unroll
      for (int k = 1; k <= 6; k++) {
        const int2 xa = at(xo[2 * k - 2], z * PL), xb = at(xo[2 * k - 1], z * PL), ya = at(yo[2 * k - 2], z * PL),
                   yb = at(yo[2 * k - 1], z * PL), za = at(me, zoff(z - k)), zb = at(me, zoff(z + k));
        fix_mad(s, a.wt[k], make_int2((xa.x + xb.x + ya.x) + (yb.x + za.x + zb.x),
                                      (xa.y + xb.y + ya.y) + (yb.y + za.y + zb.y)));
      }
      t = ku * (double)((s.hi << (FIX_LO - S_DROP)) + (s.lo >> S_DROP));
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
    mx = max(mx, abs_hw(t));
  }
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
// m <= S_MULT times: the m whose constant is closest to a double.
int weight_multiple(double h, double* ku) {
  const double hh = h * h, hl = std::fma(h, h, -hh);   // h^2 = hh + hl exactly
  int best = 1;
  double err = 1.0;
  for (int m = 1; m <= S_MULT; m++) {
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
// 4,169 points x 8 60 | 49, x 32 64 | 64, 45,025 x 1 79 | 66, x 4 80 | 87, x 32 129 | 222,
// 97,569 x 1 90 | 82, x 4 91 | 119
bool step64_wanted(const Ham& H, int w) { return step64_available(H) && (double)H.grid.n_points * w >= 1.5e5; }

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
  a.ku *= (double)(1 << S_DROP);
  a.wt[0] = m * FIX_W0;
  for (int k = 1; k <= 6; k++) a.wt[k] = m * kFixW[k - 1];
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
