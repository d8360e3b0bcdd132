// FP64 Gram matrices and rotations on the bf16 tensor cores (Cholesky-QR and Rayleigh-Ritz of
// CheFSI with FP64 blocks, arXiv 2303.00790 CheFSI paragraph).
//
// The GB300 multiplies FP64 at 1/64 of its FP32 rate (1.0 TFLOP/s) and bf16 at 1.9 PFLOP/s, so
// the products are done in integer pieces (the error-free splitting of Ozaki, Ogita, Oishi &
// Rump 2012, with fixed-point digits): every value is rounded to a 56-bit integer in units set
// by its column (Gram) or row (rotation),
//   x = 2^(E - 55) sum_i d_i 256^i,  i = 0..6,  -128 <= d_i <= 128,  |x| < 2^E,
// the digits are exact in bf16, and the 34 products d_i d_j with i + j >= 5 are accumulated per
// i + j in eight FP32 accumulators in tensor memory.  Over a chain of 128 terms every
// accumulator stays below 7 * 2^14 * 128 < 2^24, so all its sums are exact integers; after
// each chain they are added into 64-bit integers (hi: i + j = 9..12, lo: 5..8) in registers.
// What is rounded: the 56-bit conversion (2^-56 of the column's or row's largest value) and one
// conversion of the integer sum to FP64; the dropped products are below 2^-61.  (With i + j >= 6
// only, 28 products, their 2^-54 was the largest error: 1.4 to 6 times the FP64 kernels'.)
//
// gram:   C (FP64) = scale * A^T B; columns scaled by their largest element; the CTAs' integer
//         sums meet in integer atomics, so C does not depend on their order.
// rotate: out = A Q; columns of A scaled by their largest element (folded into Q's rows), then
//         rows of A and columns of Q by theirs, so that columns of very different norms (an
//         unnormalised filtered block) keep their digits.
// A NaN, an Inf or magnitudes outside 2^+-500 in an operand set a device flag: the kernels here
// then do nothing and the CUDA-core kernels, launched behind the same flag, do the work.
//
// What bounds it: shared memory.  A 128 x 64 x 16 MMA takes 48 cycles with its operands resident
// (6 KB of them at 128 bytes per cycle; 64 and 128 cycles for N = 128 and 256, with or without
// swizzle) and ~70 here, where the copies add 1.3 KB per MMA and the chains wait for their
// drain; the tensor core would need 32.  More or finer pipeline stages changed nothing.  The
// drain of 8192 x 8 accumulators every 128 terms (16 % of the time) is not overlapped, because
// the eight accumulators of 64 columns fill tensor memory.
// Measured at 234,489 rows x 850 columns: Gram 8.1 ms and triangular rotation 8.6 ms (~0.9
// PFLOP/s of bf16 products) plus 2.0 ms for maxima and digits; the CUDA-core FP64 kernels took
// ~450 and ~480 ms.  Errors against exact sums, relative to |a||b|, rms: Gram 45,025 x 100 4e-19
// (FP64 kernel 3e-18), rotation 30,000 x 850 x 850 relative 9e-17 (1e-15), with column norms over
// eight decades 2.4e-16 (3.2e-16).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "kscf_internal.h"
#include "tc_util.cuh"

namespace kscf {

namespace {

constexpr int F_DIG = 7;                       // digits per value
constexpr int F_MIN = 5;                       // products d_i d_j with i + j >= F_MIN are kept
constexpr int F_LEV = 2 * F_DIG - 1 - F_MIN;   // accumulators, one per i + j
constexpr int F_TM = 128, F_TN = 64, F_TK = 32;
constexpr int F_BLK = 128 * F_TK;              // elements of one digit of an operand block
constexpr int F_CHAIN = 4;                     // K blocks per exact chain (128 terms)
constexpr int F_STAGES = 2;
constexpr int F_A_BYTES = F_DIG * F_BLK * 2;   // 56 KB
constexpr int F_B_BYTES = F_A_BYTES / 2;       // 28 KB
constexpr int F_STAGE_BYTES = F_A_BYTES + F_B_BYTES;
constexpr int F_SMEM = F_STAGES * F_STAGE_BYTES + 1024 + 256;
constexpr int F_THREADS = 320;                 // producer, MMA, eight epilogue warps
constexpr int F_EXP_LO = 1023 - 500, F_EXP_HI = 1023 + 500;   // accepted biased exponents of maxima

__device__ unsigned int g_f64_status;   // 0 ok, else a wait timed out
__device__ __forceinline__ bool f_wait(uint64_t* bar, uint32_t parity) { return mbar_wait(bar, parity, &g_f64_status); }

__device__ __forceinline__ uint32_t abs_hw(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ int bexp(double v) {   // biased exponent, denormals as 1
  return max(1, (int)(abs_hw(v) >> 20));
}

// round(v 2^(sh - exponent of v's last bit)): v's 53-bit significand shifted left by sh (<= 2) or
// right with rounding, signed.  Integer instructions only.
__device__ __forceinline__ long long shifted(double v, int sh) {
  const long long b = __double_as_longlong(v);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if ((b >> 52) & 0x7ff) m |= 1ull << 52;
  unsigned long long t;
  if (sh >= 0) {
    t = m << min(sh, 2);
  } else {
    const int n = min(-sh, 60);
    t = (m + (1ull << (n - 1))) >> n;
  }
  return b < 0 ? -(long long)t : (long long)t;
}

// the digits of eight integers as seven 16-byte rows of a core matrix.  With 128 added at
// every digit but the top one, the digits are the bytes less 128: 128 + (byte & 127) is the
// bf16 0x4300 | (byte & 127), from which 128 (bit 7 set) or 256 is subtracted, two digits per
// packed instruction.  The top digit, -128 .. 128, goes through an FP32 magic number.
__device__ __forceinline__ void store_digits(const long long (&x)[8], __nv_bfloat16* dst) {
  uint32_t yl[8];
  int yh[8];
#pragma unroll
  for (int u = 0; u < 8; u++) {
    const long long y = x[u] + 0x0000808080808080ll;
    yl[u] = (uint32_t)y;
    yh[u] = (int)(y >> 32);
  }
#pragma unroll
  for (int s = 0; s < F_DIG; s++) {
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (s < F_DIG - 1) {
        const int q = s & 3;
        const uint32_t sel = q | (q << 4) | ((4 + q) << 8) | ((4 + q) << 12);
        const uint32_t v = s < 4 ? __byte_perm(yl[2 * u], yl[2 * u + 1], sel)
                                 : __byte_perm((uint32_t)yh[2 * u], (uint32_t)yh[2 * u + 1], sel);
        const uint32_t m = (v & 0x007f007fu) | 0x43004300u, c = (~v & 0x00800080u) | 0x43004300u;
        const __nv_bfloat162 d = __hsub2(*(const __nv_bfloat162*)&m, *(const __nv_bfloat162*)&c);
        w[u] = *(const uint32_t*)&d;
      } else {
        const float f0 = __int_as_float(0x4b400000 + (yh[2 * u] >> 16)) - 12582912.0f;
        const float f1 = __int_as_float(0x4b400000 + (yh[2 * u + 1] >> 16)) - 12582912.0f;
        w[u] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
      }
    }
    *(uint4*)(dst + s * F_BLK) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// operand storage: block (mb, kb) of 128 MN rows x 32 K holds its seven digits one after the
// other; inside a digit element (r, c) sits at (r/8)*256 + (c/8)*64 + (r%8)*8 + (c%8)
__device__ __forceinline__ int64_t blk_off(int64_t mb, int nkb, int kb) { return (mb * nkb + kb) * (F_DIG * F_BLK); }
__device__ __forceinline__ int tile_off(int r, int c) { return (r >> 3) * 256 + (c >> 3) * 64 + (r & 7) * 8 + (c & 7); }

// cmax[i] = max high word (sign cleared) of column i over the rows (mapped); *flag |= 1 when a
// column's maximum is outside the accepted range (a column of zeros is accepted) -- by the
// check kernel below, after all rows are in
__global__ void __launch_bounds__(256) col_max_kernel(const double* __restrict__ X, int64_t ld, int64_t rows, int nc,
                                                      const int32_t* __restrict__ rowmap, uint32_t* __restrict__ cmax) {
  __shared__ uint32_t red[8][32];
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), wy = threadIdx.x >> 5;
  uint32_t m = 0;
  if (i < nc) {
    const int64_t step = (int64_t)gridDim.y * 8;
    int64_t r = (int64_t)blockIdx.y * 8 + wy;
    for (; r + 3 * step < rows; r += 4 * step) {
      uint32_t h[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int64_t q = r + u * step;
        h[u] = abs_hw(X[(rowmap ? (int64_t)rowmap[q] : q) * ld + i]);
      }
      m = max(m, max(max(h[0], h[1]), max(h[2], h[3])));
    }
    for (; r < rows; r += step) m = max(m, abs_hw(X[(rowmap ? (int64_t)rowmap[r] : r) * ld + i]));
  }
  red[wy][threadIdx.x & 31] = m;
  __syncthreads();
  if (wy == 0 && i < nc) {
#pragma unroll
    for (int u = 1; u < 8; u++) m = max(m, red[u][threadIdx.x]);
    atomicMax(cmax + i, m);
  }
}

__device__ __forceinline__ bool bad_max(uint32_t hw) {
  const int e = (int)(hw >> 20);
  return e > F_EXP_HI || (e < F_EXP_LO && hw != 0);
}

__global__ void check_max_kernel(const uint32_t* a, int na, const uint32_t* b, int nb, int* flag) {
  bool bad = false;
  for (int i = threadIdx.x; i < na; i += blockDim.x) bad |= bad_max(a[i]);
  for (int i = threadIdx.x; i < nb; i += blockDim.x) bad |= bad_max(b[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) *flag = 1;
}

// qmax[j] = max high word of column j of Q (column-major).  One warp per column.
__global__ void __launch_bounds__(256) q_max_kernel(const double* __restrict__ Q, int64_t ldq, int kin, int kout,
                                                    uint32_t* __restrict__ qmax) {
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (j >= kout) return;
  uint32_t m = 0;
  for (int i = threadIdx.x & 31; i < kin; i += 32) m = max(m, abs_hw(__ldg(Q + i + (int64_t)j * ldq)));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) qmax[j] = m;
}

// Gram operand: MN = columns, K = rows r0 .. r0 + nr (mapped).  One CTA per (128 x 32) block, a
// thread per (column, 8-row group).
__global__ void __launch_bounds__(256) digits_T_kernel(const double* __restrict__ X, int64_t ld, int64_t r0, int nr,
                                                       int nc, int nkb, const int32_t* __restrict__ rowmap,
                                                       const uint32_t* __restrict__ cmax, const int* __restrict__ flag,
                                                       __nv_bfloat16* __restrict__ D) {
  if (*flag) return;
  const int kb = blockIdx.x, mb = blockIdx.y;
  __nv_bfloat16* base = D + blk_off(mb, nkb, kb);
  const int i = threadIdx.x & 127, gi = mb * 128 + i;
  const int e = gi < nc ? (int)(cmax[gi] >> 20) : 0;
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int ko = (threadIdx.x >> 7) + 2 * h;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int gr = kb * F_TK + ko * 8 + u;
      v[u] = 0.0;
      if (gi < nc && gr < nr) v[u] = X[(rowmap ? (int64_t)rowmap[r0 + gr] : r0 + gr) * ld + gi];
    }
    long long x[8];
#pragma unroll
    for (int u = 0; u < 8; u++) x[u] = shifted(v[u], bexp(v[u]) - e + 2);
    store_digits(x, base + tile_off(i, ko * 8));
  }
}

// Rotation A operand: MN = rows, K = columns; columns are taken relative to their maximum
// (cmax), the row's largest relative exponent is its unit (rexp, <= 0; a row of zeros gets
// -4096).  Rows nr .. of the last block are zero.  Eight rows per CTA: a warp per row finds the
// units; then a lane has 8 columns of one of the eight rows, so that eight lanes store the 128
// bytes of a core matrix.  HBM bound (8 B read, 14 B written per value); a warp per row for the
// digits too, storing 16 bytes of every line, and zero tests in FP64 (64 cycles each) took
// 2.11 ms at 234,489 x 850, this takes 1.00 ms.
__global__ void __launch_bounds__(256) digits_N_kernel(const double* __restrict__ X, int64_t ld, int64_t nr, int nc,
                                                       int nkb, const int32_t* __restrict__ rowmap,
                                                       const uint32_t* __restrict__ cmax, const int* __restrict__ flag,
                                                       __nv_bfloat16* __restrict__ D, int* __restrict__ rexp) {
  __shared__ int s_unit[8];
  if (*flag) return;
  const int64_t r0 = (int64_t)blockIdx.x * 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool vec = (ld & 1) == 0 && ((uintptr_t)X & 15) == 0;
  // eight values of row r from column c on (zeros outside)
  auto load8 = [&](const double* row, bool live, int c, double* v) {
    if (live && vec && c + 8 <= nc) {
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const double2 t = __ldg((const double2*)(row + c) + u);
        v[2 * u] = t.x;
        v[2 * u + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; u++) v[u] = live && c + u < nc ? row[c + u] : 0.0;
    }
  };
  auto row_of = [&](int64_t r) { return X + (r < nr ? (rowmap ? (int64_t)rowmap[r] : r) : 0) * ld; };
  auto rel = [&](double v, int c) { return bexp(v) - (c < nc ? (int)(cmax[c] >> 20) : 0); };
  auto nonzero = [](double v) { return (__double_as_longlong(v) << 1) != 0; };
  {
    const int64_t r = r0 + warp;
    const double* row = row_of(r);
    int m = -4096;
    for (int c = lane * 8; c < nc; c += 256) {
      double v[8];
      load8(row, r < nr, c, v);
#pragma unroll
      for (int u = 0; u < 8; u++)
        if (nonzero(v[u])) m = max(m, rel(v[u], c + u));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) {
      rexp[r] = m;
      s_unit[warp] = m;
    }
  }
  __syncthreads();
  const int64_t r = r0 + (lane & 7);
  const double* row = row_of(r);
  const int m = s_unit[lane & 7];
  const int64_t mb = r0 >> 7;
  for (int c = (warp * 4 + (lane >> 3)) * 8; c < nkb * F_TK; c += 256) {
    double v[8];
    load8(row, r < nr, c, v);
    long long x[8];
#pragma unroll
    for (int u = 0; u < 8; u++) x[u] = nonzero(v[u]) ? shifted(v[u], rel(v[u], c + u) - m + 2) : 0;
    store_digits(x, D + blk_off(mb, nkb, c / F_TK) + tile_off((int)(r & 127), c % F_TK));
  }
}

// Rotation B operand: MN = output columns j, K = i, of Q[i + j ldq] 2^(exponent of column i of
// A); qexp[j] = the column's largest exponent of that product.  One warp per column.
__global__ void __launch_bounds__(256) digits_Q_kernel(const double* __restrict__ Q, int64_t ldq, int kin, int kout,
                                                       int nkb, const uint32_t* __restrict__ cmax,
                                                       const int* __restrict__ flag, __nv_bfloat16* __restrict__ D,
                                                       int* __restrict__ qexp) {
  if (*flag) return;
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const double* col = Q + (int64_t)j * ldq;
  auto at = [&](int i) { return j < kout && i < kin ? __ldg(col + i) : 0.0; };
  auto ex = [&](double v, int i) { return bexp(v) + (i < kin ? (int)(cmax[i] >> 20) : 0); };
  int m = -4096;
  for (int i = lane; i < kin; i += 32) {
    const double v = at(i);
    if (v != 0.0) m = max(m, ex(v, i));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) qexp[j] = m;
  for (int c = lane * 8; c < nkb * F_TK; c += 256) {
    long long x[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const double v = at(c + u);
      x[u] = v != 0.0 ? shifted(v, ex(v, c + u) - m + 2) : 0;
    }
    store_digits(x, D + blk_off(j >> 7, nkb, c / F_TK) + tile_off(j & 127, c % F_TK));
  }
}

// four columns of all eight accumulators (columns t, t + F_TN, ...)
__device__ __forceinline__ void tmem_ld_levels(uint32_t t, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4, %5, %6, %7}, [%33];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8, %9, %10, %11}, [%34];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12, %13, %14, %15}, [%35];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16, %17, %18, %19}, [%36];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20, %21, %22, %23}, [%37];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24, %25, %26, %27}, [%38];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28, %29, %30, %31}, [%39];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]),
        "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
        "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]),
        "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]),
        "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]),
        "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]),
        "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]),
        "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31])
      : "r"(t + 0 * F_TN), "r"(t + 1 * F_TN), "r"(t + 2 * F_TN), "r"(t + 3 * F_TN), "r"(t + 4 * F_TN), "r"(t + 5 * F_TN), "r"(t + 6 * F_TN), "r"(t + 7 * F_TN)
      : "memory");
}

// (hi 2^32 + lo) 2^ex, rounded to nearest (64 leading bits kept); integer instructions only
__device__ __forceinline__ double digits_value(long long hi, long long lo, int ex) {
  const __int128 v = ((__int128)hi << 32) + lo;
  if (v == 0) return 0.0;
  unsigned __int128 m = v < 0 ? -(unsigned __int128)v : (unsigned __int128)v;
  const unsigned long long mh = (unsigned long long)(m >> 64);
  const int z = mh ? __clzll((long long)mh) : 64 + __clzll((long long)(unsigned long long)m);
  const unsigned long long t = (unsigned long long)((m << z) >> 64);   // leading one at bit 63
  unsigned long long f = (t >> 11) + ((t >> 10) & 1);                    // 53 bits, round half up
  int e = ex + 127 - z;                                                  // exponent of the leading one
  if (f >> 53) {
    f >>= 1;
    e++;
  }
  double r;
  if (e >= -1022 && e <= 1023)
    r = __longlong_as_double((long long)((f & 0xfffffffffffffull) | ((unsigned long long)(e + 1023) << 52)));
  else
    r = scalbn((double)f, e - 52);
  return v < 0 ? -r : r;
}

struct F64Args {
  const __nv_bfloat16 *A, *B;   // digits
  int nkb;                      // K blocks of the operands
  int m_tiles, n_tiles;         // tiles of 128 (M) and 64 (N)
  int m, n;                     // valid output rows (gram) and columns
  const int* flag;
  // gram
  int kb_per_cta;               // multiple of F_CHAIN
  int symmetric;                // tiles above the diagonal only
  unsigned long long* acc;      // (hi, lo) integer sums, m x n column-major
  // rotate
  int upper;                    // Q upper triangular: tile nt needs K < (nt + 1) 64
  const int *rexp, *qexp;
  int64_t rows;
  const int32_t* rowmap;
  double* out;
  int64_t ldo;
};

// One kernel for both: GRAM handles the tile blockIdx.x over the K range blockIdx.y and adds
// to C atomically; else persistent over tiles (N fastest, so that CTAs sharing an A panel run
// side by side), whole K, rows of out written.
template <bool GRAM>
__global__ void __launch_bounds__(F_THREADS, 1) f64_mma_kernel(F64Args p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + F_STAGES * F_STAGE_BYTES);
  uint64_t* empty = full + F_STAGES;
  uint64_t* tfull = empty + F_STAGES;
  uint64_t* tempty = tfull + 1;
  uint32_t* tmem_slot = (uint32_t*)(tempty + 1);
  if (*p.flag) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntiles = p.m_tiles * p.n_tiles;
  // tile t -> (mt, nt), K blocks [kb0, kb0 + nk)
  auto tile = [&](int t, int* mt, int* nt, int* kb0, int* nk) {
    if (GRAM) {
      *mt = t % p.m_tiles;
      *nt = t / p.m_tiles;
      *kb0 = blockIdx.y * p.kb_per_cta;
      *nk = min(p.nkb, *kb0 + p.kb_per_cta) - *kb0;
      if (p.symmetric && *nt * F_TN + F_TN - 1 < *mt * F_TM) *nk = 0;
    } else {
      *nt = t % p.n_tiles;
      *mt = t / p.n_tiles;
      *kb0 = 0;
      *nk = p.upper ? min(p.nkb, (*nt + 1) * (F_TN / F_TK)) : p.nkb;
    }
  };
  const int t0 = blockIdx.x, tstep = GRAM ? ntiles : gridDim.x;
  if (GRAM) {
    int mt, nt, kb0, nk;
    tile(t0, &mt, &nt, &kb0, &nk);
    if (nk <= 0) return;
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < F_STAGES; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int t = t0; t < ntiles && ok; t += tstep) {
        int mt, nt, kb0, nk;
        tile(t, &mt, &nt, &kb0, &nk);
        for (int k = 0; k < nk; k++, g++) {
          const int s = g % F_STAGES;
          if (g >= F_STAGES && !f_wait(&empty[s], ((g / F_STAGES) - 1) & 1)) {
            ok = false;
            break;
          }
          uint8_t* sa = smem + s * F_STAGE_BYTES;
          uint8_t* sb = sa + F_A_BYTES;
          mbar_expect_tx(&full[s], F_STAGE_BYTES);
          bulk_g2s(sa, p.A + blk_off(mt, p.nkb, kb0 + k), F_A_BYTES, &full[s]);
          // B: the 64 rows of this tile inside their 128-row block, one copy per digit
          const __nv_bfloat16* b = p.B + blk_off(nt >> 1, p.nkb, kb0 + k) + (nt & 1) * (F_BLK / 2);
          for (int d = 0; d < F_DIG; d++) bulk_g2s(sb + d * F_BLK, b + d * F_BLK, F_BLK, &full[s]);
        }
      }
      // the copies of the last stages issued have landed before the CTA can exit
      for (int q = max(0, g - F_STAGES); q < g; q++) f_wait(&full[q % F_STAGES], (q / F_STAGES) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int g = 0, ch = 0;
      bool ok = true;
      constexpr uint32_t idesc = idesc_n(F_TN);
      for (int t = t0; t < ntiles && ok; t += tstep) {
        int mt, nt, kb0, nk;
        tile(t, &mt, &nt, &kb0, &nk);
        for (int k0 = 0; k0 < nk && ok; k0 += F_CHAIN, ch++) {
          if (ch >= 1 && !f_wait(tempty, (ch - 1) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int k1 = min(nk, k0 + F_CHAIN);
          for (int k = k0; k < k1; k++, g++) {
            const int s = g % F_STAGES;
            ok = f_wait(&full[s], (g / F_STAGES) & 1);
            if (!ok) break;
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + s * F_STAGE_BYTES);
            const uint32_t sb = sa + F_A_BYTES;
#pragma unroll
            for (int kk = 0; kk < F_TK / 16; kk++) {
#pragma unroll
              for (int i = 0; i < F_DIG; i++) {
                const uint64_t ad = smem_desc(sa + i * F_BLK * 2 + kk * 256, 128, 512);
#pragma unroll
                for (int j = (i < F_MIN ? F_MIN - i : 0); j < F_DIG; j++) {
                  const uint64_t bd = smem_desc(sb + j * F_BLK + kk * 256, 128, 512);
                  // accumulator i + j - 5; the first product into it in this order has i = 0 or j = 6
                  mma_bf16(tmem + (i + j - F_MIN) * F_TN, ad, bd, idesc,
                           (k > k0 || kk > 0 || (i > 0 && j < F_DIG - 1)) ? 1u : 0u);
                }
              }
            }
            mma_commit(&empty[s]);
          }
          mma_commit(tfull);
        }
      }
    }
  } else {
    // epilogue warps 2..9: TMEM lane quadrant warp % 4, columns (warp - 2) / 4 * 32 ..
    const int q = warp & 3, h = (warp - 2) >> 2;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + h * 32;
    int ch = 0;
    bool ok = true;
    for (int t = t0; t < ntiles && ok; t += tstep) {
      int mt, nt, kb0, nk;
      tile(t, &mt, &nt, &kb0, &nk);
      long long hi[32], lo[32];
#pragma unroll
      for (int c = 0; c < 32; c++) hi[c] = lo[c] = 0;
      for (int k0 = 0; k0 < nk; k0 += F_CHAIN, ch++) {
        ok = __all_sync(0xffffffffu, f_wait(tfull, ch & 1));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < 32; c0 += 4) {
          uint32_t r[32];
          tmem_ld_levels(tbase + c0, r);
#pragma unroll
          for (int c = 0; c < 4; c++) {
            int a[F_LEV];
#pragma unroll
            for (int l = 0; l < F_LEV; l++) a[l] = __float2int_rn(__uint_as_float(r[l * 4 + c]));
            // |a[7 - q]| <= (q + 1) 2^21: the 32-bit combinations stay below 2^31
            const int top = a[7] * 256 + a[6], mid = a[5] * 256 + a[4];
            hi[c0 + c] += (long long)top * 65536 + mid;
            lo[c0 + c] += ((long long)a[3] * 256 + a[2]) * 65536 + ((long long)a[1] * 256 + a[0]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tempty)) : "memory");
      }
      if (!ok) break;
      const int i = mt * F_TM + q * 32 + lane, j0 = nt * F_TN + h * 32;
      if (GRAM) {
        if (i < p.m) {
#pragma unroll
          for (int c = 0; c < 32; c++) {
            const int j = j0 + c;
            if (j < p.n && (!p.symmetric || j >= i)) {
              unsigned long long* s2 = p.acc + 2 * (i + (int64_t)j * p.m);
              atomicAdd(s2, (unsigned long long)hi[c]);
              atomicAdd(s2 + 1, (unsigned long long)lo[c]);
            }
          }
        }
      } else if (i < p.rows) {
        double* o = p.out + (p.rowmap ? (int64_t)__ldg(p.rowmap + i) : (int64_t)i) * p.ldo;
        const int er = p.rexp[i] - 2 * 1077 + 40;
        const bool vec = (p.ldo & 1) == 0 && ((uintptr_t)p.out & 15) == 0;
#pragma unroll
        for (int c = 0; c < 32; c += 2) {
          const int j = j0 + c;
          if (j >= p.n) break;
          const double v0 = digits_value(hi[c], lo[c], er + __ldg(p.qexp + j));
          const double v1 = j + 1 < p.n ? digits_value(hi[c + 1], lo[c + 1], er + __ldg(p.qexp + j + 1)) : 0.0;
          if (vec && j + 1 < p.n) {
            *(double2*)(o + j) = make_double2(v0, v1);
          } else {
            o[j] = v0;
            if (j + 1 < p.n) o[j + 1] = v1;
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// C = scale * the integer sums (exact, so the result does not depend on the order of the CTAs);
// symmetric: the lower triangle from the upper one.  Units 2^(e_a - 1077) and 2^(e_b - 1077) of
// the two columns, lo in 256^5 of them.
__global__ void __launch_bounds__(256) gram_out_kernel(const unsigned long long* __restrict__ acc, int m, int n,
                                                       const uint32_t* __restrict__ ca, const uint32_t* __restrict__ cb,
                                                       double scale, int symmetric, const int* __restrict__ flag,
                                                       double* __restrict__ C, int64_t ldc) {
  if (*flag) return;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)m * n) return;
  const int j = (int)(idx / m), i = (int)(idx - (int64_t)j * m);
  const bool low = symmetric && i > j;
  const int a = low ? j : i, b = low ? i : j;   // the element computed
  const longlong2 s = *(const longlong2*)(acc + 2 * (a + (int64_t)b * m));
  const int ex = (int)(ca[a] >> 20) + (int)(cb[b] >> 20) - 2 * 1077 + 40;
  C[i + (int64_t)j * ldc] = scale * digits_value(s.x, s.y, ex);
}

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
size_t digit_bytes(int64_t mn, int64_t k) { return (size_t)(cdiv(mn, 128) * cdiv(k, F_TK)) * F_DIG * F_BLK * 2; }

constexpr int64_t F_CHUNK_MAX = 131072;                 // rows per launch
constexpr int64_t F_ROWS_MAX = (int64_t)1 << 22;        // |lo| < 2^47.4 per 128 rows: 64-bit sums hold
constexpr size_t F_PIECE_BUDGET = (size_t)1 << 30;      // bytes of digits per Gram launch or row panel of kscf_rotate

// flag, column maxima, integer sums (n_b: columns with digits of their own, 0 for a Gram of
// one operand; n: columns of the result)
size_t gram_head(int m, int n_b, int n) {
  return kscf_align256((size_t)(m + n_b) * 4) + 256 + kscf_align256((size_t)m * n * 16);
}
size_t gram_bytes(int64_t chunk, int m, int n) {
  return gram_head(m, n, n) + kscf_align256(digit_bytes(m, chunk)) + kscf_align256(digit_bytes(n, chunk)) + 512;
}
// largest row chunk (multiple of 128, at most F_CHUNK_MAX) whose digits fit
int64_t gram_chunk(int64_t rows, int m, int n_b, int n, size_t bytes) {
  const size_t head = gram_head(m, n_b, n) + 512, per = digit_bytes(m, 128) + digit_bytes(n_b, 128);
  if (bytes < head + per) return 0;
  return std::min<int64_t>(std::min<int64_t>((int64_t)((bytes - head) / per) * 128, F_CHUNK_MAX), cdiv(rows, 128) * 128);
}
size_t rot_head(int64_t rows, int kin, int kout) {
  return kscf_align256((size_t)kin * 4) + kscf_align256((size_t)cdiv(rows, 128) * 128 * 4) +
         kscf_align256((size_t)cdiv(kout, 128) * 128 * 4) + 256;
}

cudaError_t sm_count(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  return e;
}

cudaError_t col_max(const double* X, int64_t ld, int64_t rows, int nc, const int32_t* rowmap, uint32_t* cmax, int sms,
                    cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(cmax, 0, (size_t)nc * 4, st);
  if (e != cudaSuccess) return e;
  const int gx = (int)cdiv(nc, 32);
  const int gy = (int)std::max<int64_t>(1, std::min<int64_t>(cdiv(rows, 256), cdiv(8 * sms, gx)));
  col_max_kernel<<<dim3(gx, gy), 256, 0, st>>>(X, ld, rows, nc, rowmap, cmax), count_launch();
  return cudaGetLastError();
}

}  // namespace

// Where the lines lie (measured, us, this path | CUDA-core kernels): Gram 128 rows x 1 column 43 | 141,
// 128 x 100 53 | 144, 512 x 8 44 | 546, 4,169 x 8 44 | 899, 45,025 x 16 90 | 1087, 234,489 x 2 282 | 2078
// -- everywhere, since the CUDA-core kernel walks up to 1024 rows in one FP64 chain; less than a tile of
// 128 rows stays there (100 rows: 122).  Rotation 45,025
// rows x 16 107 | 88, x 24 116 | 168, 4,169 x 32 61 | 41, x 100 69 | 127, 234,489 x 8 362 | 405.
bool gram_f64tc_wanted(int64_t rows) { return rows >= 128 && rows <= F_ROWS_MAX; }
bool rotate_f64tc_wanted(int64_t rows, int kin, int kout) {
  return (int64_t)kin * kout >= 24 * 24 && (double)rows * kin * kout >= 5e6 && rows <= F_ROWS_MAX;
}

size_t gram_f64tc_work_bytes(int64_t rows, int m, int n) {
  const size_t per = digit_bytes(m, 128) + digit_bytes(n, 128);
  const int64_t want = std::max<int64_t>(1, (int64_t)(F_PIECE_BUDGET / per)) * 128;
  return gram_bytes(std::min<int64_t>(std::min<int64_t>(want, F_CHUNK_MAX), cdiv(rows, 128) * 128), m, n);
}
// Rotation of 234,489 x 850 by 850 x 850: one panel of 2.7 GB 15.06 ms, three of 1 GiB 15.23, eleven of 256 MiB 15.62
int64_t rotate_f64tc_panel(int64_t rows, int kin) {
  const int64_t fit = (int64_t)(F_PIECE_BUDGET / digit_bytes(128, kin)) * 128;
  return std::min<int64_t>(std::max<int64_t>(fit, 128), rows);
}
size_t rotate_f64tc_work_bytes(int64_t rows, int kin, int kout) {
  return rot_head(rows, kin, kout) + kscf_align256(digit_bytes(rows, kin)) + kscf_align256(digit_bytes(kout, kin));
}
bool gram_f64tc_fits(int64_t rows, int m, int n, bool same, size_t bytes) {
  return gram_chunk(rows, m, same ? 0 : n, n, bytes) >= std::min<int64_t>(cdiv(rows, 128) * 128, 4096);
}

cudaError_t launch_gram_f64tc(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t rows, int m, int n,
                              double scale, double* C, int64_t ldc, void* work, size_t work_bytes, bool symmetric,
                              const int32_t* rowmap, cudaStream_t st) {
  const bool same = A == B && lda == ldb && m == n;
  const bool sym = same || (symmetric && m == n);
  const int64_t chunk = gram_chunk(rows, m, same ? 0 : n, n, work_bytes);
  if (chunk < 128) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  char* w = (char*)work;
  int* flag = (int*)w;
  uint32_t* ca = (uint32_t*)(w + 256);
  uint32_t* cb = same ? ca : ca + m;
  unsigned long long* acc = (unsigned long long*)(w + 256 + kscf_align256((size_t)(m + (same ? 0 : n)) * 4));
  w += gram_head(m, same ? 0 : n, n);
  __nv_bfloat16* Ad = (__nv_bfloat16*)w;
  __nv_bfloat16* Bd = same ? Ad : (__nv_bfloat16*)(w + kscf_align256(digit_bytes(m, chunk)));
  if ((e = cudaMemset2DAsync(C, (size_t)ldc * 8, 0, (size_t)m * 8, n, st)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(flag, 0, 4, st)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(acc, 0, (size_t)m * n * 16, st)) != cudaSuccess) return e;
  if ((e = col_max(A, lda, rows, m, rowmap, ca, sms, st)) != cudaSuccess) return e;
  if (!same && (e = col_max(B, ldb, rows, n, rowmap, cb, sms, st)) != cudaSuccess) return e;
  check_max_kernel<<<1, 256, 0, st>>>(ca, m, cb, same ? 0 : n, flag), count_launch();
  if ((e = cudaFuncSetAttribute(f64_mma_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM)) !=
      cudaSuccess)
    return e;
  F64Args a = {};
  a.A = Ad;
  a.B = Bd;
  a.m_tiles = (int)cdiv(m, F_TM);
  a.n_tiles = (int)cdiv(n, F_TN);
  a.m = m;
  a.n = n;
  a.flag = flag;
  a.symmetric = sym ? 1 : 0;
  a.acc = acc;
  int active = 0;
  for (int nt = 0; nt < a.n_tiles; nt++)
    for (int mt = 0; mt < a.m_tiles; mt++) active += !(sym && nt * F_TN + F_TN - 1 < mt * F_TM);
  for (int64_t r0 = 0; r0 < rows; r0 += chunk) {
    const int nr = (int)std::min<int64_t>(chunk, rows - r0);
    a.nkb = (int)cdiv(nr, F_TK);
    digits_T_kernel<<<dim3(a.nkb, a.m_tiles), 256, 0, st>>>(A, lda, r0, nr, m, a.nkb, rowmap, ca, flag, Ad),
        count_launch();
    if (!same)
      digits_T_kernel<<<dim3(a.nkb, (unsigned)cdiv(n, 128)), 256, 0, st>>>(B, ldb, r0, nr, n, a.nkb, rowmap, cb, flag,
                                                                           Bd),
          count_launch();
    // split K so that the active CTAs fill whole waves of one CTA per SM
    int best_ks = 1;
    double best = -1.0;
    const int max_ks = (int)cdiv(a.nkb, F_CHAIN);
    for (int cand = 1; cand <= max_ks && (cand == 1 || (int64_t)active * cand <= 8 * sms); cand++) {
      const int kpc = (int)(cdiv(cdiv(a.nkb, cand), F_CHAIN) * F_CHAIN), real = (int)cdiv(a.nkb, kpc);
      const int64_t ctas = (int64_t)active * real;
      // time of the last wave's CTAs, in K blocks, with a fixed cost of 4 K blocks per CTA
      const double time = (double)cdiv(ctas, sms) * (kpc + 4);
      const double score = 1.0 / time;
      if (score > best * (1 + 1e-9)) {
        best = score;
        best_ks = cand;
      }
    }
    a.kb_per_cta = (int)(cdiv(cdiv(a.nkb, best_ks), F_CHAIN) * F_CHAIN);
    f64_mma_kernel<true><<<dim3(a.m_tiles * a.n_tiles, (unsigned)cdiv(a.nkb, a.kb_per_cta)), F_THREADS, F_SMEM, st>>>(a),
        count_launch();
  }
  e = launch_gram_native(A, lda, B, ldb, rows, m, n, KSCF_F64, scale, C, ldc, true, st, rowmap, flag);
  if (e != cudaSuccess) return e;
  gram_out_kernel<<<(unsigned)cdiv((int64_t)m * n, 256), 256, 0, st>>>(acc, m, n, ca, cb, scale, sym ? 1 : 0, flag, C,
                                                                       ldc),
      count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rotate_f64tc(const double* A, int64_t lda, const double* Q, int64_t ldq, int64_t rows, int kin,
                                int kout, bool upper, double* out, int64_t ldo, void* work, size_t work_bytes,
                                const int32_t* rowmap, int64_t max_rows, bool reuse_q, const int** flag_out,
                                cudaStream_t st) {
  if (work_bytes < rotate_f64tc_work_bytes(rows, kin, kout)) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  char* w = (char*)work;
  auto take = [&](size_t b) {
    char* q = w;
    w += kscf_align256(b);
    return q;
  };
  int* flag = (int*)take(256);
  uint32_t* ca = (uint32_t*)take((size_t)kin * 4);
  // what the row panels of one product share comes first
  int* qexp = (int*)take((size_t)cdiv(kout, 128) * 128 * 4);
  __nv_bfloat16* Bd = (__nv_bfloat16*)take(digit_bytes(kout, kin));
  int* rexp = (int*)take((size_t)cdiv(rows, 128) * 128 * 4);
  __nv_bfloat16* Ad = (__nv_bfloat16*)take(digit_bytes(rows, kin));
  *flag_out = flag;
  if (max_rows > 0) {
    if ((e = cudaMemsetAsync(flag, 0, 4, st)) != cudaSuccess) return e;
    if ((e = col_max(A, lda, max_rows, kin, rowmap, ca, sms, st)) != cudaSuccess) return e;
  }
  const int nkb = (int)cdiv(kin, F_TK);
  if (!reuse_q) {
    // Q's columns: their maxima only tell whether all elements are finite and in range
    q_max_kernel<<<(unsigned)cdiv(kout, 8), 256, 0, st>>>(Q, ldq, kin, kout, (uint32_t*)qexp), count_launch();
    check_max_kernel<<<1, 256, 0, st>>>(ca, kin, (const uint32_t*)qexp, kout, flag), count_launch();
    digits_Q_kernel<<<(unsigned)(cdiv(kout, 128) * 16), 256, 0, st>>>(Q, ldq, kin, kout, nkb, ca, flag, Bd, qexp),
        count_launch();
  }
  digits_N_kernel<<<(unsigned)(cdiv(rows, 128) * 16), 256, 0, st>>>(A, lda, rows, kin, nkb, rowmap, ca, flag, Ad, rexp),
      count_launch();
  if ((e = cudaFuncSetAttribute(f64_mma_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM)) !=
      cudaSuccess)
    return e;
  F64Args a = {};
  a.A = Ad;
  a.B = Bd;
  a.nkb = nkb;
  a.m_tiles = (int)cdiv(rows, F_TM);
  a.n_tiles = (int)cdiv(kout, F_TN);
  a.m = (int)rows;
  a.n = kout;
  a.flag = flag;
  a.upper = upper ? 1 : 0;
  a.rexp = rexp;
  a.qexp = qexp;
  a.rows = rows;
  a.rowmap = rowmap;
  a.out = out;
  a.ldo = ldo;
  const int ntiles = a.m_tiles * a.n_tiles;
  f64_mma_kernel<false><<<std::min(ntiles, sms), F_THREADS, F_SMEM, st>>>(a), count_launch();
  return cudaGetLastError();
}

cudaError_t f64tc_status(bool reset, unsigned int* status) {
  cudaError_t e = cudaMemcpyFromSymbol(status, g_f64_status, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  if (reset && *status) {
    unsigned int z = 0;
    e = cudaMemcpyToSymbol(g_f64_status, &z, sizeof(unsigned int));
  }
  return e;
}

}  // namespace kscf
