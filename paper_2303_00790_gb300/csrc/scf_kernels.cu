// Kernels of the self-consistent field loop (arXiv 2303.00790, Computational details:
// Kohn-Sham DFT in the LDA, SCF stopped on the self-consistent residual error):
//   - Gaussian atomic valence densities (start of the SCF),
//   - LDA exchange-correlation: Slater exchange + Perdew-Zunger 1981 correlation,
//   - Hartree potential: -Lap_h V_H = 4 pi rho by conjugate gradients in FP64 on the
//     Hilbert-brick grid, with the values the order-12 stencil needs outside the sphere
//     taken from the multipole expansion (monopole, dipole, quadrupole) of rho,
//   - residual V_out - V_in, SRE and the energy integrals,
//   - Anderson mixing of the input potential.
// All arithmetic is FP64.  Reductions are deterministic: every block writes one partial
// sum per value, and consumers add the partials in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>

#include "cg_offsets.cuh"
#include "fixlap.cuh"
#include "fp64.cuh"
#include "kscf_internal.h"
#include "scf_internal.h"

namespace kscf {

static inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Sum of p[0..nb) in a fixed order; every lane of the calling warp gets the same value
// (a butterfly of commutative additions).
__device__ __forceinline__ double warp_sum_partials(const double* __restrict__ p, int nb) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int i = lane; i < nb; i += 32) s += p[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Block-wide sum of NV values per thread; thread 0 writes part[v * gridDim.x + blockIdx.x].
template <int NV>
__device__ __forceinline__ void block_partials(double (&v)[NV], double* __restrict__ part) {
  __shared__ double sh[NV][kScfThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; q++) {
    double s = v[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sh[q][warp] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NV; q++) {
      double s = 0.0;
      for (int w = 0; w < kScfThreads / 32; w++) s += sh[q][w];
      part[q * gridDim.x + blockIdx.x] = s;
    }
  }
}

// out[v] = sum_b part[v * nb + b]  (one block; warp w handles values w, w + 8, ...)
__global__ void finalize_partials_kernel(const double* __restrict__ part, int nb, int nv, double* __restrict__ out) {
  const int warp = threadIdx.x >> 5;
  for (int v = warp; v < nv; v += blockDim.x >> 5) {
    const double s = warp_sum_partials(part + (int64_t)v * nb, nb);
    if ((threadIdx.x & 31) == 0) out[v] = s;
  }
}

cudaError_t launch_finalize_partials(const double* part, int nb, int nv, double* out, cudaStream_t st) {
  finalize_partials_kernel<<<1, 256, 0, st>>>(part, nb, nv, out), count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Starting density: rho(p) = sum_a Z_a / (pi^{3/2} r_a^3) exp(-|p - R_a|^2 / r_a^2).
// atoms: 5 doubles each (x, y, z, Z_valence, r_a); rel: h * (i, j, k) of every slot.
// Bound by the FP64 pipe.  What depends on the atom alone is formed once per CTA; the quotient by
// r_a^2 is a product with its reciprocal corrected by the remainder; and where every lane's
// exponential is below 2^-86 while its sum is above 2^-32 of the atom's prefactor, the term
// is below half a unit of the sum and left out.  45,025 points, 71 atoms: 555 -> 362 us.
__global__ void atomic_density_kernel(const double* __restrict__ rel, double cx, double cy, double cz,
                                      const uint8_t* __restrict__ mask, const double* __restrict__ atoms,
                                      int n_atoms, int64_t n, double* __restrict__ rho) {
  __shared__ double sat[128 * 7];   // x, y, z, prefactor, r_a^2, 1 / r_a^2, 2^-32 of the prefactor
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = s < n && mask[s];
  double px = 0, py = 0, pz = 0;
  if (live) {
    px = cx + rel[3 * s];
    py = cy + rel[3 * s + 1];
    pz = cz + rel[3 * s + 2];
  }
  double acc = 0.0;
  for (int a0 = 0; a0 < n_atoms; a0 += 128) {
    const int na = min(128, n_atoms - a0);
    __syncthreads();
    for (int q = threadIdx.x; q < na; q += blockDim.x) {
      const double* at = atoms + (int64_t)(a0 + q) * 5;
      const double ra = at[4];
      for (int c = 0; c < 3; c++) sat[7 * q + c] = at[c];
      sat[7 * q + 3] = at[3] / (5.568327996831707845 * ra * ra * ra);
      sat[7 * q + 4] = ra * ra;
      sat[7 * q + 5] = 1.0 / (ra * ra);
      sat[7 * q + 6] = fabs(sat[7 * q + 3]) * 0x1.0p-32;
    }
    __syncthreads();
    if (live) {
      for (int a = 0; a < na; a++) {
        const double* at = sat + 7 * a;
        const double dx = px - at[0], dy = py - at[1], dz = pz - at[2];
        const double d2 = dx * dx + dy * dy + dz * dz;
        const double q0 = d2 * at[5];
        // (bits of values >= 0 compare like the values; 60 > 86 ln 2)
        const bool small = __double_as_longlong(q0) > __double_as_longlong(60.0) &&
                           __double_as_longlong(acc) > __double_as_longlong(at[6]);
        if (__all_sync(__activemask(), small)) continue;
        const bool finite = __double_as_longlong(q0) < __double_as_longlong(0x1p1000);
        acc += at[3] * exp(finite ? -fma(fma(-q0, at[4], d2), at[5], q0) : -q0);
      }
    }
  }
  if (s < n) rho[s] = live ? acc : 0.0;
}

cudaError_t launch_atomic_density(const Ham& H, const double* rel, const double* atoms, int n_atoms, double* rho,
                                  cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  atomic_density_kernel<<<nblk(n, 128), 128, 0, st>>>(rel, H.grid.center[0], H.grid.center[1], H.grid.center[2],
                                                     H.d_mask, atoms, n_atoms, n, rho), count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// LDA (unpolarised, Hartree units).  Slater exchange eps_x = -3/4 (3 rho/pi)^{1/3},
// v_x = 4/3 eps_x.  Perdew-Zunger 1981 fit of the Ceperley-Alder correlation energy,
// rs = (3/(4 pi rho))^{1/3}:
//   rs >= 1: eps_c = gamma / (1 + beta1 sqrt(rs) + beta2 rs),
//            v_c = eps_c (1 + 7/6 beta1 sqrt(rs) + 4/3 beta2 rs) / (1 + beta1 sqrt(rs) + beta2 rs)
//   rs <  1: eps_c = A ln rs + B + C rs ln rs + D rs,
//            v_c = A ln rs + (B - A/3) + 2/3 C rs ln rs + (2D - C)/3 rs
// gamma = -0.1423, beta1 = 1.0529, beta2 = 0.3334, A = 0.0311, B = -0.048, C = 0.0020,
// D = -0.0116.  Densities at or below 1e-14 give zero.
__global__ void lda_kernel(const double* __restrict__ rho, const uint8_t* __restrict__ mask, int64_t n,
                           double* __restrict__ eps, double* __restrict__ vxc) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  double e = 0.0, v = 0.0;
  const double r = rho[s];
  if (mask[s] && r > 1e-14) {
    const double pi = 3.14159265358979323846;
    const double rs = cbrt(3.0 / (4.0 * pi * r));
    const double ex = -0.75 * cbrt(3.0 * r / pi);
    const double vx = (4.0 / 3.0) * ex;
    double ec, vc;
    if (rs >= 1.0) {
      const double sq = sqrt(rs);
      const double den = 1.0 + 1.0529 * sq + 0.3334 * rs;
      ec = -0.1423 / den;
      vc = ec * (1.0 + 7.0 / 6.0 * 1.0529 * sq + 4.0 / 3.0 * 0.3334 * rs) / den;
    } else {
      const double ln = log(rs);
      ec = 0.0311 * ln + (-0.048) + 0.0020 * rs * ln + (-0.0116) * rs;
      vc = 0.0311 * ln + (-0.048 - 0.0311 / 3.0) + 2.0 / 3.0 * 0.0020 * rs * ln + (2.0 * (-0.0116) - 0.0020) / 3.0 * rs;
    }
    e = ex + ec;
    v = vx + vc;
  }
  if (eps) eps[s] = e;
  vxc[s] = v;
}

cudaError_t launch_lda(const Ham& H, const double* rho, double* eps, double* vxc, cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  lda_kernel<<<nblk(n, 256), 256, 0, st>>>(rho, H.d_mask, n, eps, vxc), count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// CG operator A x = -Lap_h x + shift x on the domain (zero outside: padding slots of x
// hold zero and missing bricks read as zero): shift 0 for the Poisson problem, q0^2 for
// the Kerker preconditioner.  cw[k] = -w_k / h^2 (k = 0..6); the centre term uses
// 3 cw[0].  One thread per slot.
struct LapArgs {
  const int32_t* nbr;
  const uint8_t* mask;
  double cw[7];
  double shift;
  int64_t n;
};

template <int B>
__device__ __forceinline__ double lap_at(const LapArgs& a, const double* __restrict__ x, int64_t s) {
  constexpr int B3 = B * B * B;
  const int64_t brick = s / B3;
  const int li = (int)(s - brick * B3);
  const int l[3] = {li % B, (li / B) % B, li / (B * B)};
  const int stride[3] = {1, B, B * B};
  double acc = (3.0 * a.cw[0] + a.shift) * x[s];
#pragma unroll
  for (int ax = 0; ax < 3; ax++) {
#pragma unroll
    for (int k = 1; k <= 6; k++) {
      double pair = 0.0;
#pragma unroll
      for (int sg = -1; sg <= 1; sg += 2) {
        const int nn = l[ax] + sg * k;
        if (nn >= 0 && nn < B) {
          pair += x[s + (int64_t)sg * k * stride[ax]];
        } else {
          const int nb = a.nbr[brick * 6 + 2 * ax + (sg > 0 ? 1 : 0)];
          if (nb >= 0) pair += x[(int64_t)nb * B3 + li + (sg * k - sg * B) * stride[ax]];
        }
      }
      acc += a.cw[k] * pair;
    }
  }
  return acc;
}

// b = 4 pi rho + sum over the ghost points g of the slot: w_g V_ghost[g]; partial b.b
__global__ void __launch_bounds__(kScfThreads) poisson_rhs_kernel(const double* __restrict__ rho,
                                                                  const uint8_t* __restrict__ mask,
                                                                  const int64_t* __restrict__ gptr,
                                                                  const int32_t* __restrict__ gidx,
                                                                  const double* __restrict__ gw,
                                                                  const double* __restrict__ vghost, int64_t n,
                                                                  double* __restrict__ b, double* __restrict__ part) {
  double acc[1] = {0.0};
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    double v = 0.0;
    if (mask[s]) {
      v = 4.0 * 3.14159265358979323846 * rho[s];
      for (int64_t e = gptr[s]; e < gptr[s + 1]; e++) v += gw[e] * vghost[gidx[e]];
    }
    b[s] = v;
    acc[0] += v * v;
  }
  block_partials<1>(acc, part);
}

// r = b - A x, p = r, partial r.r  (x is the starting guess; padding rows set to zero)
template <int B>
__global__ void __launch_bounds__(kScfThreads) cg_init_kernel(LapArgs a, double* __restrict__ x,
                                                              const double* __restrict__ b, double* __restrict__ r,
                                                              double* __restrict__ p, double* __restrict__ part_rr) {
  double acc[1] = {0.0};
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < a.n; s += (int64_t)gridDim.x * blockDim.x) {
    double rv = 0.0;
    if (a.mask[s]) rv = b[s] - lap_at<B>(a, x, s);
    r[s] = rv;
    p[s] = rv;
    acc[0] += rv * rv;
  }
  block_partials<1>(acc, part_rr);
}

// ---------------------------------------------------------------------------
// The conjugate gradients in one cooperative launch (one CTA per SM, the domain points in
// contiguous shares, two bounded grid barriers per iteration):
//   q = A r + beta q, p = r + beta p, p.q | x += alpha p, r -= alpha q, r.r
// (q = A p by the recurrence of Chronopoulos & Gear 1989, so that the only neighbour values
// read are those of r, which are ready at the barrier of r.r.)  A r reads r as 58-bit fixed
// point (fixlap.cuh), whose exponent comes from max|r| and max|q| of the reductions before.
// What bounds an iteration is latency: at 45,025 points (one per thread; cycles) the star takes
// 1,500, the CTA's sums 2 x 950, the barriers 2 x 2,500, the partial sums from L2 2 x 1,500, the
// divisions 1,400, the update 500; at 234,489 points the star 11,500 (loads, and 5 of the 10
// FP64 instructions per point at 64 cycles per warp) and the update 2,700.  Up to 4 points per
// thread the vectors stay in registers; larger grids (NPT = 0) keep them in global memory.  Three
// launches per iteration with the star in FP64 and every warp adding the 304 partials two or
// three times took 89 us at 234,489 points and 67 us at 45,025; this kernel takes 14.0 us and
// 7.1 us (Hartree solve of the 2.2 nm cluster, 368 iterations: 32.7 -> 5.18 ms).
constexpr int kCgThreads = 512;   // most threads of a CTA

struct CgArgs {
  LapArgs a;
  const int32_t* live;      // domain slots
  int64_t n_live;
  double lap_unit;          // -FIX_SUM_UNIT / (831600 h^2)
  int has_shift;            // a.shift is not zero
  double *x, *r, *p, *q;
  int2* rf;                 // r in fixed point, zero in padding slots
  const double* rr_in;      // partial sums of r.r at entry
  int n_rr;
  const double* part_bb;
  int n_bb;
  double rtol2;
  double* part;             // 2 x grid partial sums: p.q, r.r
  uint32_t* hmax;           // 2 x grid maxima of the high words of |q|, |r|
  double* state;            // out: r.r, b.b, beta (in unless first)
  int* iters;               // += iterations done
  unsigned* bar;            // arrival counter, zero at launch
  int* status;              // 1: a barrier wait gave up
  long long spin_limit;
  int max_iters;
  int first;                // p, q start from zero
};

// Grid barrier as in the eigensolver's tridiagonalisation: release arrivals on a monotonic
// counter, acquire polls, bounded by spin_limit clock cycles.
// cg_arrive is called after a CTA barrier that follows the other threads' stores; work that no
// other CTA reads can stand between it and cg_wait.
__device__ __forceinline__ void cg_arrive(const CgArgs& c) {
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(c.bar) : "memory");
}
__device__ bool cg_wait(const CgArgs& c, unsigned target, int* s_ok) {
  if (threadIdx.x == 0) {
    int ok = 1;
    const long long t0 = clock64();
    for (unsigned tries = 1;; tries++) {
      unsigned n;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(c.bar) : "memory");
      if (n >= target) break;
      // (the status word is another trip to L2: not between every two looks at the counter)
      if (tries % 32 == 0 && (*(volatile int*)c.status != 0 || clock64() - t0 > c.spin_limit)) {
        atomicExch(c.status, 1);
        ok = 0;
        break;
      }
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}
__device__ __forceinline__ bool cg_barrier(const CgArgs& c, unsigned target, int* s_ok) {
  cg_arrive(c);
  return cg_wait(c, target, s_ok);
}

// CTA sum of v and maximum of m into *sum and *mx (global, thread 0): two levels of warp sums.
// red, shm: kCgThreads / 32.
__device__ __forceinline__ void cg_reduce(double v, uint32_t m, double* red, uint32_t* shm, double* sum,
                                          uint32_t* mx) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) {
    red[warp] = v;
    shm[warp] = m;
  }
  __syncthreads();
  if (warp == 0) {
    const double s = warp_sum(lane < nw ? red[lane] : 0.0);
    const uint32_t t = __reduce_max_sync(0xffffffffu, lane < nw ? shm[lane] : 0u);
    if (lane == 0) {
      *sum = s;
      *mx = t;
    }
  }
}

// Sum of part[0..P) and maximum of mx[0..P) in one warp; the loads are issued together.
__device__ __forceinline__ double cg_collect(const double* part, const uint32_t* mx, int P, uint32_t* m_out) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  uint32_t m = 0;
  for (int b0 = 0; b0 < P; b0 += 160) {
    double v[5];
    uint32_t u[5];
#pragma unroll
    for (int q = 0; q < 5; q++) {
      const int b = b0 + 32 * q + lane;
      v[q] = b < P ? __ldcg(part + b) : 0.0;
      u[q] = b < P ? __ldcg(mx + b) : 0u;
    }
    const double t = ((v[0] + v[1]) + (v[2] + v[3])) + v[4];
    s = b0 == 0 ? t : s + t;
#pragma unroll
    for (int q = 0; q < 5; q++) m = max(m, u[q]);
  }
  *m_out = __reduce_max_sync(0xffffffffu, m);
  return warp_sum(s);
}

// v 2^k (exact) for normal v, in integer instructions where the result is normal
__device__ __forceinline__ double scale_pow2(double v, int k) {
  const long long b = __double_as_longlong(v);
  const int e = ((int)(b >> 52) & 0x7ff) + k;
  return e >= 1 && e <= 2046 ? __longlong_as_double(b + ((long long)k << 52)) : scalbn(v, k);
}

// A double at least every double whose high word (sign cleared) is hw
__device__ __forceinline__ double hw_bound(uint32_t hw) { return __hiloint2double((int)min(hw + 1, 0x7ff00000u), 0); }
__device__ __forceinline__ uint32_t abs_hw(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }

// The fixed-point field's base for the offsets of cg_offsets.cuh
template <int B>
__device__ __forceinline__ const char* cg_base(const int2* rf) {
  return (const char*)(rf - B * B * B);
}
// Face neighbours of slot s: nb[2 ax + sg] +- 8 k stride is the slot at distance k beyond the
// brick's face; a missing brick points into the zeros behind the field (kCgZeroSlots), so that
// the star needs no predicates.
template <int B, typename O>
__device__ __forceinline__ void cg_faces(const int32_t* nbr, int s, O zero, O* nb) {
  constexpr int B3 = B * B * B;
  const int brick = s / B3, li = s - brick * B3;
#pragma unroll
  for (int f = 0; f < 6; f++) nb[f] = cg_face<O, B>(__ldg(nbr + (int64_t)brick * 6 + f), li, f, zero);
}

// 831600 h^2 Lap_h of the fixed-point field (f: its cg_base) at slot s
template <int B, typename O>
__device__ __forceinline__ FixAcc cg_star(const char* f, int s, const O* nb, int nbs) {
  const int li = s & (B * B * B - 1);
  const int l[3] = {li % B, (li / B) % B, li / (B * B)};
  const int stride[3] = {1, B, B * B};
  const O own = cg_own<O, B>(s);
  FixAcc acc = {0, 0};
  fix_mad(acc, FIX_W0, *(const int2*)(f + own));
  O face[6];
#pragma unroll
  for (int q = 0; q < 6; q++) face[q] = nb[q * nbs];
#pragma unroll
  for (int k = 1; k <= 6; k++) {
    int2 v[6];
#pragma unroll
    for (int ax = 0; ax < 3; ax++) {
      const O lo = l[ax] >= k ? own : face[2 * ax], hi = l[ax] + k < B ? own : face[2 * ax + 1];
      v[2 * ax] = *(const int2*)(f + (size_t)lo - 8 * k * stride[ax]);
      v[2 * ax + 1] = *(const int2*)(f + (size_t)hi + 8 * k * stride[ax]);
    }
    fix_mad(acc, FIX_W[k - 1], make_int2((v[0].x + v[1].x + v[2].x) + (v[3].x + v[4].x + v[5].x),
                                         (v[0].y + v[1].y + v[2].y) + (v[3].y + v[4].y + v[5].y)));
  }
  return acc;
}

// O: type of the offsets into the field
template <int B, int NPT, typename O = uint32_t>
__global__ void __launch_bounds__(kCgThreads, 1) cg_kernel(CgArgs c) {
  static_assert(NPT == 0 || sizeof(O) == 4, "the vectors of a large field are not in registers");
  extern __shared__ uint32_t s_face[];   // NPT > 0: [6][NPT][threads] face neighbours of the points
  __shared__ double sh[kCgThreads / 32];
  __shared__ uint32_t shm[kCgThreads / 32];
  __shared__ double s_val[2];
  __shared__ uint32_t s_max;
  __shared__ int s_ok;
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, P = gridDim.x, cta = blockIdx.x;
  const int64_t per = (c.n_live + P - 1) / P;
  const int64_t i0 = cta * per, i1 = min(c.n_live, i0 + per);
  double* part_pq = c.part;
  double* part_rr = c.part + P;
  uint32_t* max_q = c.hmax;
  uint32_t* max_r = c.hmax + P;
  unsigned target = 0;
  const O zero = cg_zero<O>(c.a.n, kCgZeroSlots);
  constexpr int NR = NPT > 0 ? NPT : 1;
  int sv[NR];
  double xv[NR], rv[NR], pv[NR], qv[NR];
  // f(point number k of the thread, slot, x, r, p, q) over the thread's points; the vectors
  // are registers or global memory.  With registers a thread without a k-th point works on a
  // zero point behind the field (all its values stay zero), so that the points interleave
  // without branches.
  auto each = [&](auto f) {
    if constexpr (NPT > 0) {
#pragma unroll
      for (int k = 0; k < NPT; k++) f(k, sv[k], xv[k], rv[k], pv[k], qv[k]);
    } else {
      for (int64_t i = i0 + tid; i < i1; i += nt) {
        const int s = c.live[i];
        f(0, s, c.x[s], c.r[s], c.p[s], c.q[s]);
      }
    }
  };
  if constexpr (NPT > 0) {
#pragma unroll
    for (int k = 0; k < NPT; k++) {
      const int64_t i = i0 + tid + (int64_t)k * nt;
      const bool on = i < i1;
      sv[k] = on ? c.live[i] : (int)(zero / 8);
      O nb[6];
      if (on) cg_faces<B>(c.a.nbr, sv[k], zero, nb);
#pragma unroll
      for (int q = 0; q < 6; q++) s_face[(q * NPT + k) * nt + tid] = on ? nb[q] : zero + 8 * (B * B * B);
      xv[k] = on ? c.x[sv[k]] : 0.0;
      rv[k] = on ? c.r[sv[k]] : 0.0;
      pv[k] = on && !c.first ? c.p[sv[k]] : 0.0;
      qv[k] = on && !c.first ? c.q[sv[k]] : 0.0;
    }
  } else if (c.first) {
    each([&](int, int, double&, double&, double& p, double& q) { p = q = 0.0; });
  }
  // the largest |r|, r.r and b.b at entry, r in fixed point
  uint32_t mr = 0;
  each([&](int, int, double&, double& r, double&, double&) { mr = max(mr, abs_hw(r)); });
  __syncthreads();
  cg_reduce(0.0, mr, sh, shm, part_pq + cta, max_r + cta);
  if (!cg_barrier(c, target += P, &s_ok)) return;
  if (warp == 0) {
    const double rr0 = warp_sum_partials(c.rr_in, c.n_rr), bb0 = warp_sum_partials(c.part_bb, c.n_bb);
    uint32_t m;
    cg_collect(part_pq, max_r, P, &m);
    if (lane == 0) {
      s_val[0] = rr0;
      s_val[1] = bb0;
      s_max = m;
    }
  }
  __syncthreads();
  double rr = s_val[0], beta = c.first ? 0.0 : c.state[2];
  const double bb = s_val[1];
  mr = s_max;
  int e = fix_exp(mr);
  each([&](int, int s, double&, double& r, double&, double&) { c.rf[s] = fix_from(r, e); });
  __syncthreads();
  if (!cg_barrier(c, target += P, &s_ok)) return;
  const long long tol_bits = __double_as_longlong(c.rtol2 * bb);
  int it = 0;
  for (; it < c.max_iters; it++) {
    // rr < rtol^2 b.b or not finite; rr >= 0, so the bits compare like the values (FP64
    // comparisons and products in every warp, here and in sc, took 64 cycles each of its pipe)
    const long long rr_bits = __double_as_longlong(rr);
    if (rr_bits < tol_bits || rr_bits >= 0x7ff0000000000000LL) break;
    // q = A r + beta q, p = r + beta p, p.q
    const double sc = scale_pow2(c.lap_unit, e - 1022 - FIX_BITS);
    double acc = 0.0;
    uint32_t mq = 0;
    each([&](int k, int s, double&, double& r, double& p, double& q) {
      FixAcc t;
      if constexpr (NPT > 0) {
        t = cg_star<B>(cg_base<B>(c.rf), s, s_face + k * nt + tid, NPT * nt);
      } else {
        O nb[6];
        cg_faces<B>(c.a.nbr, s, zero, nb);
        t = cg_star<B>(cg_base<B>(c.rf), s, nb, 1);
      }
      const double pn = fma(beta, p, r);
      double qn = fma(sc, fix_value(t), beta * q);
      if (c.has_shift) qn = fma(c.a.shift, r, qn);
      p = pn;
      q = qn;
      acc = fma(pn, qn, acc);
      mq = max(mq, abs_hw(qn));
    });
    cg_reduce(acc, mq, sh, shm, part_pq + cta, max_q + cta);
    if (!cg_barrier(c, target += P, &s_ok)) return;
    if (warp == 0) {
      uint32_t m;
      const double pq = cg_collect(part_pq, max_q, P, &m);
      if (lane == 0) {
        const double alpha = rr / pq;
        s_val[0] = alpha;
        // |r - alpha q| <= max|r| + |alpha| max|q|
        s_max = abs_hw(fma(fabs(alpha), hw_bound(m), hw_bound(mr)));
      }
    }
    __syncthreads();
    const double alpha = s_val[0];
    e = fix_exp(s_max);
    // r -= alpha q, r.r; x += alpha p while the CTA waits for the others
    acc = 0.0;
    mr = 0;
    each([&](int, int s, double&, double& r, double&, double& q) {
      const double rn = fma(-alpha, q, r);
      r = rn;
      c.rf[s] = fix_from(rn, e);
      acc = fma(rn, rn, acc);
      mr = max(mr, abs_hw(rn));
    });
    cg_reduce(acc, mr, sh, shm, part_rr + cta, max_r + cta);
    cg_arrive(c);
    each([&](int, int, double& x, double&, double& p, double&) { x = fma(alpha, p, x); });
    if (!cg_wait(c, target += P, &s_ok)) return;
    if (warp == 0) {
      uint32_t m;
      const double t = cg_collect(part_rr, max_r, P, &m);
      if (lane == 0) {
        s_val[0] = t;
        s_val[1] = t / rr;
        s_max = m;
      }
    }
    __syncthreads();
    rr = s_val[0];
    beta = s_val[1];
    mr = s_max;
  }
  if constexpr (NPT > 0) {
#pragma unroll
    for (int k = 0; k < NPT; k++) {
      if (i0 + tid + (int64_t)k * nt >= i1) continue;
      c.x[sv[k]] = xv[k];
      c.r[sv[k]] = rv[k];
      c.p[sv[k]] = pv[k];
      c.q[sv[k]] = qv[k];
    }
  }
  if (cta == 0 && tid == 0) {
    c.state[0] = rr;
    c.state[1] = bb;
    c.state[2] = beta;
    c.iters[0] += it;
  }
}

template <int B>
static cudaError_t cg_launch(CgArgs& c, int P, cudaStream_t st) {
  const int64_t per = (c.n_live + P - 1) / P;
  const int npt = (int)((per + kCgThreads - 1) / kCgThreads);
  // the fewest threads that hold the share with npt points each, so that the warps are full
  int nt = npt <= 4 ? (int)(((per + npt - 1) / npt + 31) / 32 * 32) : kCgThreads;
  nt = std::max(nt, 128);
  const int smem = npt <= 4 ? 6 * npt * nt * (int)sizeof(int) : 0;
  const bool wide = cg_wide(c.a.n, kCgZeroSlots, B);
  const void* k = npt == 1   ? (const void*)cg_kernel<B, 1>
                  : npt == 2 ? (const void*)cg_kernel<B, 2>
                  : npt == 3 ? (const void*)cg_kernel<B, 3>
                  : npt == 4 ? (const void*)cg_kernel<B, 4>
                  : wide     ? (const void*)cg_kernel<B, 0, uint64_t>
                             : (const void*)cg_kernel<B, 0>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {&c};
  return cudaLaunchCooperativeKernel(k, dim3(P), dim3(nt), args, smem, st);
}

static LapArgs lap_args(const Ham& H, double shift) {
  LapArgs a;
  a.shift = shift;
  a.nbr = H.d_nbr;
  a.mask = H.d_mask;
  // H.stencil[k] = -1/2 w_k / h^2, so -w_k / h^2 = 2 H.stencil[k]
  for (int k = 0; k <= 6; k++) a.cw[k] = 2.0 * H.stencil[k];
  a.n = H.grid.n_slots;
  return a;
}

cudaError_t launch_poisson_rhs(const Ham& H, const double* rho, const PoissonPlan& P, double* b, double* part_bb,
                               cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  poisson_rhs_kernel<<<kScfRedBlocks, kScfThreads, 0, st>>>(rho, H.d_mask, P.d_gptr, P.d_gidx, P.d_gw, P.d_vghost,
                                                            n, b, part_bb), count_launch();
  return cudaGetLastError();
}

cudaError_t launch_cg_init(const Ham& H, double shift, double* x, const double* b, double* r, double* p,
                           double* part_rr, cudaStream_t st) {
  const LapArgs a = lap_args(H, shift);
  if (H.grid.B == 8)
    cg_init_kernel<8><<<kScfRedBlocks, kScfThreads, 0, st>>>(a, x, b, r, p, part_rr), count_launch();
  else
    cg_init_kernel<16><<<kScfRedBlocks, kScfThreads, 0, st>>>(a, x, b, r, p, part_rr), count_launch();
  return cudaGetLastError();
}

cudaError_t launch_cg(const Ham& H, double shift, const CgWork& w, double rtol, double* x, const double* rr_in,
                      int n_rr, bool first, int max_iters, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.sync, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  CgArgs c;
  c.a = lap_args(H, shift);
  c.live = H.d_live;
  c.n_live = H.n_live;
  c.lap_unit = -1.0 / (FIX_DEN * H.grid.h * H.grid.h) * FIX_SUM_UNIT;
  c.has_shift = shift != 0.0 ? 1 : 0;
  c.x = x;
  c.r = w.r;
  c.p = w.p;
  c.q = w.q;
  c.rf = (int2*)w.rf;
  c.rr_in = rr_in;
  c.n_rr = n_rr;
  c.part_bb = w.part_bb;
  c.n_bb = kScfRedBlocks;
  c.rtol2 = rtol * rtol;
  c.part = w.part;
  c.hmax = w.hmax;
  c.state = w.state;
  c.iters = w.iters;
  c.bar = w.sync;
  c.status = (int*)w.sync + 1;
  c.spin_limit = 2000000000LL;   // ~1 s
  c.max_iters = max_iters;
  c.first = first ? 1 : 0;
  // one CTA per SM; a CTA takes at least 128 points (small grids: fewer CTAs, cheaper barriers)
  const int P = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(sms, kScfRedBlocks), (H.n_live + 127) / 128));
  e = H.grid.B == 8 ? cg_launch<8>(c, P, st) : cg_launch<16>(c, P, st);
  count_launch();
  return e;
}

// b = f on the domain (0 outside); partial b.b
__global__ void __launch_bounds__(kScfThreads) rhs_copy_kernel(const double* __restrict__ f,
                                                               const uint8_t* __restrict__ mask, int64_t n,
                                                               double* __restrict__ b, double* __restrict__ part) {
  double acc[1] = {0.0};
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    const double v = mask[s] ? f[s] : 0.0;
    b[s] = v;
    acc[0] += v * v;
  }
  block_partials<1>(acc, part);
}

cudaError_t launch_rhs_copy(const Ham& H, const double* f, double* b, double* part_bb, cudaStream_t st) {
  rhs_copy_kernel<<<kScfRedBlocks, kScfThreads, 0, st>>>(f, H.d_mask, H.grid.n_slots, b, part_bb), count_launch();
  return cudaGetLastError();
}

// out = a + c b (0 outside the domain)
__global__ void lincomb_kernel(const uint8_t* __restrict__ mask, const double* __restrict__ a,
                               const double* __restrict__ b, double c, int64_t n, double* __restrict__ out) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n) out[s] = mask[s] ? a[s] + c * b[s] : 0.0;
}

cudaError_t launch_lincomb(const Ham& H, const double* a, const double* b, double c, double* out, cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  lincomb_kernel<<<nblk(n, 256), 256, 0, st>>>(H.d_mask, a, b, c, n, out), count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Multipoles of rho about the grid centre (x = h (i, j, k)); partials of
// q = sum rho, p_i = sum rho x_i, S_ij = sum rho x_i x_j  (10 values; times h^3 later).
__global__ void __launch_bounds__(kScfThreads) multipole_kernel(const double* __restrict__ rho,
                                                                const double* __restrict__ rel, int64_t n,
                                                                double* __restrict__ part) {
  double v[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    const double r = rho[s];
    if (r == 0.0) continue;
    const double x = rel[3 * s], y = rel[3 * s + 1], z = rel[3 * s + 2];
    v[0] += r;
    v[1] += r * x;
    v[2] += r * y;
    v[3] += r * z;
    v[4] += r * x * x;
    v[5] += r * y * y;
    v[6] += r * z * z;
    v[7] += r * x * y;
    v[8] += r * x * z;
    v[9] += r * y * z;
  }
  block_partials<10>(v, part);
}

// V at each ghost point t (relative to the centre):
//   q/|t| + p.t/|t|^3 + 1/2 t^T Q t / |t|^5,  Q_ij = 3 S_ij - delta_ij tr S  (all times h^3)
__global__ void ghost_potential_kernel(const double* __restrict__ mom, double h3, const double* __restrict__ grel,
                                       int64_t ng, double* __restrict__ vghost) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= ng) return;
  const double q = h3 * mom[0];
  const double px = h3 * mom[1], py = h3 * mom[2], pz = h3 * mom[3];
  const double tr = mom[4] + mom[5] + mom[6];
  const double Qxx = h3 * (3.0 * mom[4] - tr), Qyy = h3 * (3.0 * mom[5] - tr), Qzz = h3 * (3.0 * mom[6] - tr);
  const double Qxy = h3 * 3.0 * mom[7], Qxz = h3 * 3.0 * mom[8], Qyz = h3 * 3.0 * mom[9];
  const double x = grel[3 * g], y = grel[3 * g + 1], z = grel[3 * g + 2];
  const double r2 = x * x + y * y + z * z;
  const double r = sqrt(r2);
  const double quad = Qxx * x * x + Qyy * y * y + Qzz * z * z + 2.0 * (Qxy * x * y + Qxz * x * z + Qyz * y * z);
  vghost[g] = q / r + (px * x + py * y + pz * z) / (r2 * r) + 0.5 * quad / (r2 * r2 * r);
}

cudaError_t launch_ghost_values(const Ham& H, const double* rho, const double* rel, const PoissonPlan& P,
                                double* part, double* mom, cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  multipole_kernel<<<kScfRedBlocks, kScfThreads, 0, st>>>(rho, rel, n, part), count_launch();
  cudaError_t e = launch_finalize_partials(part, kScfRedBlocks, 10, mom, st);
  if (e != cudaSuccess) return e;
  const double h3 = H.grid.h * H.grid.h * H.grid.h;
  if (P.n_ghost > 0)
    ghost_potential_kernel<<<nblk(P.n_ghost, 256), 256, 0, st>>>(mom, h3, P.d_grel, P.n_ghost, P.d_vghost),
        count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Residual and energy integrals:
//   f = V_out - V_in with V_out = V_ion + V_H + V_xc (zero outside the domain)
//   partials of  rho f^2,  rho (V_in - V_ion),  rho V_H,  rho eps_xc,  rho
__global__ void __launch_bounds__(kScfThreads) residual_kernel(const uint8_t* __restrict__ mask,
                                                               const double* __restrict__ rho,
                                                               const double* __restrict__ v_in,
                                                               const double* __restrict__ v_ion,
                                                               const double* __restrict__ vh,
                                                               const double* __restrict__ vxc,
                                                               const double* __restrict__ eps, int64_t n,
                                                               double* __restrict__ f, double* __restrict__ part) {
  double v[5] = {0, 0, 0, 0, 0};
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    double fv = 0.0;
    if (mask[s]) {
      const double r = rho[s];
      fv = (v_ion[s] + vh[s] + vxc[s]) - v_in[s];
      v[0] += r * fv * fv;
      v[1] += r * (v_in[s] - v_ion[s]);
      v[2] += r * vh[s];
      v[3] += r * eps[s];
      v[4] += r;
    }
    f[s] = fv;
  }
  block_partials<5>(v, part);
}

cudaError_t launch_residual(const Ham& H, const double* rho, const double* v_in, const double* v_ion, const double* vh,
                            const double* vxc, const double* eps, double* f, double* part, double* out5,
                            cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  residual_kernel<<<kScfRedBlocks, kScfThreads, 0, st>>>(H.d_mask, rho, v_in, v_ion, vh, vxc, eps, n, f, part),
      count_launch();
  return launch_finalize_partials(part, kScfRedBlocks, 5, out5, st);
}

// v = a + b + c (masked)
__global__ void sum3_kernel(const uint8_t* __restrict__ mask, const double* __restrict__ a,
                            const double* __restrict__ b, const double* __restrict__ c, int64_t n,
                            double* __restrict__ out) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n) out[s] = mask[s] ? a[s] + b[s] + c[s] : 0.0;
}

cudaError_t launch_sum3(const Ham& H, const double* a, const double* b, const double* c, double* out,
                        cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  sum3_kernel<<<nblk(n, 256), 256, 0, st>>>(H.d_mask, a, b, c, n, out), count_launch();
  return cudaGetLastError();
}

// out = a + b (masked)
__global__ void add2_kernel(const uint8_t* __restrict__ mask, const double* __restrict__ a,
                            const double* __restrict__ b, int64_t n, double* __restrict__ out) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n) out[s] = mask[s] ? a[s] + b[s] : 0.0;
}

cudaError_t launch_add2(const Ham& H, const double* a, const double* b, double* out, cudaStream_t st) {
  const int64_t n = H.grid.n_slots;
  add2_kernel<<<nblk(n, 256), 256, 0, st>>>(H.d_mask, a, b, n, out), count_launch();
  return cudaGetLastError();
}

// Column inner products in FP64: part[j * gridDim.x + b] = this block's share of
// sum_r A[r][j] B[r][j] (B = A: column sums of squares).
template <typename T>
__global__ void __launch_bounds__(kScfThreads) col_dot_kernel(const T* __restrict__ A, int64_t lda,
                                                              const T* __restrict__ B, int64_t ldb, int64_t rows,
                                                              int k, double* __restrict__ part) {
  const int64_t per = (rows + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = (int64_t)blockIdx.x * per;
  const int64_t r1 = r0 + per < rows ? r0 + per : rows;
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    double a0 = 0.0, a1 = 0.0;
    int64_t r = r0;
    for (; r + 1 < r1; r += 2) {
      a0 += (double)A[r * lda + j] * (double)B[r * ldb + j];
      a1 += (double)A[(r + 1) * lda + j] * (double)B[(r + 1) * ldb + j];
    }
    if (r < r1) a0 += (double)A[r * lda + j] * (double)B[r * ldb + j];
    part[(int64_t)j * gridDim.x + blockIdx.x] = a0 + a1;
  }
}

// part[j * gridDim.x + b] = this block's share of sum_r (HX[r][j] - lam[j] X[r][j])^2  (FP64)
template <typename T>
__global__ void __launch_bounds__(kScfThreads) col_resid_kernel(const T* __restrict__ X, const T* __restrict__ HX,
                                                                int64_t ld, int64_t rows, int k,
                                                                const double* __restrict__ lam,
                                                                double* __restrict__ part) {
  const int64_t per = (rows + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = (int64_t)blockIdx.x * per;
  const int64_t r1 = r0 + per < rows ? r0 + per : rows;
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    const double l = lam[j];
    double a = 0.0;
    for (int64_t r = r0; r < r1; r++) {
      const double d = (double)HX[r * ld + j] - l * (double)X[r * ld + j];
      a += d * d;
    }
    part[(int64_t)j * gridDim.x + blockIdx.x] = a;
  }
}

cudaError_t launch_col_dot(const void* A, int64_t lda, const void* B, int64_t ldb, int64_t rows, int k, int dtype,
                           double* part, double* out, cudaStream_t st) {
  if (dtype == KSCF_F64)
    col_dot_kernel<double><<<kScfRedBlocks, kScfThreads, 0, st>>>((const double*)A, lda, (const double*)B, ldb, rows,
                                                                  k, part), count_launch();
  else
    col_dot_kernel<float><<<kScfRedBlocks, kScfThreads, 0, st>>>((const float*)A, lda, (const float*)B, ldb, rows, k,
                                                                 part), count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_finalize_partials(part, kScfRedBlocks, k, out, st);
}

cudaError_t launch_col_sumsq(const void* X, int64_t ld, int64_t rows, int k, int dtype, double* part, double* out,
                             cudaStream_t st) {
  return launch_col_dot(X, ld, X, ld, rows, k, dtype, part, out, st);
}

cudaError_t launch_col_resid(const double* X, const double* HX, int64_t ld, int64_t rows, int k, const double* lam,
                             double* part, double* out, cudaStream_t st) {
  return launch_col_resid_t(X, HX, ld, rows, k, KSCF_F64, lam, part, out, st);
}

cudaError_t launch_col_resid_t(const void* X, const void* HX, int64_t ld, int64_t rows, int k, int dtype,
                               const double* lam, double* part, double* out, cudaStream_t st) {
  if (dtype == KSCF_F64)
    col_resid_kernel<double><<<kScfRedBlocks, kScfThreads, 0, st>>>((const double*)X, (const double*)HX, ld, rows, k,
                                                                    lam, part), count_launch();
  else
    col_resid_kernel<float><<<kScfRedBlocks, kScfThreads, 0, st>>>((const float*)X, (const float*)HX, ld, rows, k,
                                                                   lam, part), count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_finalize_partials(part, kScfRedBlocks, k, out, st);
}

// dst[r][j] = (double) src[r][j]  (FP32 -> FP64), r < rows, j < k
__global__ void widen_kernel(const float* __restrict__ src, int64_t lds, double* __restrict__ dst, int64_t ldd,
                             int64_t rows, int k) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= rows * k) return;
  const int64_t r = idx / k;
  const int j = (int)(idx - r * k);
  dst[r * ldd + j] = (double)src[r * lds + j];
}

cudaError_t launch_widen(const float* src, int64_t lds, double* dst, int64_t ldd, int64_t rows, int k,
                         cudaStream_t st) {
  widen_kernel<<<nblk(rows * k, 256), 256, 0, st>>>(src, lds, dst, ldd, rows, k), count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Anderson mixing.
// New history column: dV = V_in - V_prev, dF = F - F_prev (and dPF = PF - PF_prev when
// the residual is preconditioned); then V_prev = V_in, F_prev = F, PF_prev = PF.
__global__ void anderson_push_kernel(int64_t n, const double* __restrict__ v_in, const double* __restrict__ f,
                                     const double* __restrict__ pf, double* __restrict__ v_prev,
                                     double* __restrict__ f_prev, double* __restrict__ pf_prev,
                                     double* __restrict__ dv, double* __restrict__ df, double* __restrict__ dpf,
                                     int have_prev) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const double vi = v_in[s], fi = f[s];
  if (have_prev) {
    dv[s] = vi - v_prev[s];
    df[s] = fi - f_prev[s];
  }
  v_prev[s] = vi;
  f_prev[s] = fi;
  if (pf) {
    const double pi = pf[s];
    if (have_prev) dpf[s] = pi - pf_prev[s];
    pf_prev[s] = pi;
  }
}

cudaError_t launch_anderson_push(int64_t n, const double* v_in, const double* f, const double* pf, double* v_prev,
                                 double* f_prev, double* pf_prev, double* dv, double* df, double* dpf, bool have_prev,
                                 cudaStream_t st) {
  anderson_push_kernel<<<nblk(n, 256), 256, 0, st>>>(n, v_in, f, pf, v_prev, f_prev, pf_prev, dv, df, dpf,
                                                     have_prev ? 1 : 0), count_launch();
  return cudaGetLastError();
}

// Partials of dF_i . dF_j (i <= j, packed row-major upper) and dF_i . F, i, j < m
// (the columns in the order given by cols).
__global__ void __launch_bounds__(kScfThreads) anderson_gram_kernel(AndersonCols cols, const double* __restrict__ df,
                                                                    const double* __restrict__ f, int64_t n,
                                                                    double* __restrict__ part) {
  constexpr int NV = kAndersonMax * (kAndersonMax + 1) / 2 + kAndersonMax;
  double v[NV];
#pragma unroll
  for (int q = 0; q < NV; q++) v[q] = 0.0;
  const int m = cols.m;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    double x[kAndersonMax];
#pragma unroll
    for (int i = 0; i < kAndersonMax; i++) x[i] = i < m ? df[(int64_t)cols.idx[i] * n + s] : 0.0;
    const double fv = f[s];
    int q = 0;
#pragma unroll
    for (int i = 0; i < kAndersonMax; i++) {
#pragma unroll
      for (int j = i; j < kAndersonMax; j++) v[q++] += x[i] * x[j];
    }
#pragma unroll
    for (int i = 0; i < kAndersonMax; i++) v[q++] += x[i] * fv;
  }
  block_partials<NV>(v, part);
}

cudaError_t launch_anderson_gram(const AndersonCols& cols, const double* df, const double* f, int64_t n,
                                 double* part, double* out, cudaStream_t st) {
  constexpr int NV = kAndersonMax * (kAndersonMax + 1) / 2 + kAndersonMax;
  anderson_gram_kernel<<<kScfRedBlocks, kScfThreads, 0, st>>>(cols, df, f, n, part), count_launch();
  return launch_finalize_partials(part, kScfRedBlocks, NV, out, st);
}

// V_next = V_in + alpha PF - sum_j g_j (dV_j + alpha dPF_j)   (in place on v; PF = F and
// dPF = dF without a preconditioner)
__global__ void anderson_update_kernel(AndersonCols cols, double alpha, const uint8_t* __restrict__ mask, int64_t n,
                                       const double* __restrict__ dv, const double* __restrict__ df,
                                       const double* __restrict__ f, double* __restrict__ v) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  if (!mask[s]) {
    v[s] = 0.0;
    return;
  }
  double nv = v[s] + alpha * f[s];
  for (int j = 0; j < cols.m; j++) {
    const int64_t o = (int64_t)cols.idx[j] * n + s;
    nv -= cols.g[j] * (dv[o] + alpha * df[o]);
  }
  v[s] = nv;
}

cudaError_t launch_anderson_update(const Ham& H, const AndersonCols& cols, double alpha, const double* dv,
                                   const double* dpf, const double* pf, double* v, cudaStream_t st) {
  const double* df = dpf;
  const double* f = pf;
  const int64_t n = H.grid.n_slots;
  anderson_update_kernel<<<nblk(n, 256), 256, 0, st>>>(cols, alpha, H.d_mask, n, dv, df, f, v), count_launch();
  return cudaGetLastError();
}

// row lex(s) of D_out / t_out for every domain slot s: the slot's descriptors and
// dV = V_in - V_start (training data of the learned start)
__global__ void training_rows_kernel(const float* __restrict__ D, const double* __restrict__ v_in,
                                     const double* __restrict__ v_start, const int64_t* __restrict__ lex,
                                     int64_t n_slots, float* __restrict__ D_out, float* __restrict__ t_out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t s = t >> 5;
  const int j = (int)(t & 31);
  if (s >= n_slots) return;
  const int64_t p = lex[s];
  if (p < 0) return;
  D_out[p * KSCF_MLP_N_IN + j] = D[s * KSCF_MLP_N_IN + j];
  if (j == 0) t_out[p] = (float)(v_in[s] - v_start[s]);
}

cudaError_t launch_training_rows(const Ham& H, const float* D, const double* v_in, const double* v_start, float* D_out,
                                 float* t_out, cudaStream_t st) {
  const int64_t n = H.grid.n_slots * 32;
  training_rows_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(D, v_in, v_start, H.d_lex, H.grid.n_slots, D_out,
                                                                     t_out);
  count_launch();
  return cudaGetLastError();
}

}  // namespace kscf
