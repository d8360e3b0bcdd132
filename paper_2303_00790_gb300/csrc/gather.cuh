// Projections of a column block on the Kleinman-Bylander projectors:
//   coef[(a*4+l)*cld + v] = E_l h^3 sum over atom a's entries e of chi_l(e) Y(slot_e, v), v < w,
// and 0 for w <= v < zpad.  Element (slot s, column v) of Y sits at
//   Y[(v >> cw_log) * cs + s * ld + (v & (2^cw_log - 1))]:
// slot-major rows (cw_log = 30) or chunk-major copies.
//
// One CTA per atom and CL * VW columns; CL lanes read the columns of an entry's row (VW each, one
// vector load), the other lanes of the warp and the other warps take other entries, four in
// flight per lane, and their sums meet in shared memory.  What bounds it is latency: an entry
// costs a dependent pair of loads (slot, row), ~500 entries per atom.  CL = 32 reads each slot
// and chi once per 32 * VW columns; CL = 8 has 32 instead of 8 entry streams per CTA and a
// quarter of the columns, which is better as long as the wide CTAs do not fill the SMs: FP32, 35
// atoms x 64 columns 12 us against 40, 353 atoms x 850 columns 15.34 against 15.43 ms per
// 12-step filter; FP64, 353 x 850 102.8 against 102.1 ms, 35 x 100 2.37 against 2.63 ms per
// 10-step filter, one atom x 8 columns 14 us against ~25.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

namespace kscf {

// CTAs of the wide variant from which on it is taken
constexpr int64_t GATHER_WIDE_CTAS = 2000;

template <typename T, int VW>
struct GatherVec {
  T v[VW];
};

template <typename T>
struct GatherArgs {
  const T* Y;
  int64_t cs, ld;
  int cw_log, w, zpad;
  int64_t cld;
  const int64_t* aptr;
  const int64_t* aslot;
  const T* achi;
  const double* energy;
  T* coef;
};

template <typename T, int VW, int CL>
__global__ void __launch_bounds__(256) kb_gather_kernel(GatherArgs<T> a) {
  constexpr int SUB = 32 / CL, STREAMS = 8 * SUB, U = 4;
  const int at = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cl = lane % CL, stream = warp * SUB + lane / CL;
  const int col = (blockIdx.y * CL + cl) * VW;
  T acc[4][VW];
#pragma unroll
  for (int l = 0; l < 4; l++)
#pragma unroll
    for (int q = 0; q < VW; q++) acc[l][q] = T(0);
  if (col < a.w) {
    const T* y0 = a.Y + (int64_t)(col >> a.cw_log) * a.cs + (col & ((1 << a.cw_log) - 1));
    const int64_t e1 = __ldg(a.aptr + at + 1);
    // VW > 1: the row holds whole vectors (chunk-major copies are padded to their chunk width)
    auto row = [&](int64_t s) {
      GatherVec<T, VW> y;
      const T* p = y0 + s * a.ld;
      if constexpr (VW * sizeof(T) == 16) {
        *(float4*)&y = __ldg((const float4*)p);
      } else {
#pragma unroll
        for (int q = 0; q < VW; q++) y.v[q] = __ldg(p + q);
      }
      return y;
    };
    auto add = [&](int64_t e, const GatherVec<T, VW>& y) {
      GatherVec<T, 4> c;
      if constexpr (sizeof(T) == 4) {
        *(float4*)&c = __ldg((const float4*)(a.achi + 4 * e));
      } else {
        *(double2*)&c.v[0] = __ldg((const double2*)(a.achi + 4 * e));
        *(double2*)&c.v[2] = __ldg((const double2*)(a.achi + 4 * e) + 1);
      }
#pragma unroll
      for (int l = 0; l < 4; l++)
#pragma unroll
        for (int q = 0; q < VW; q++) acc[l][q] = fma(c.v[l], y.v[q], acc[l][q]);
    };
    int64_t e = __ldg(a.aptr + at) + stream;
    for (; e + (U - 1) * STREAMS < e1; e += U * STREAMS) {
      int64_t s[U];
#pragma unroll
      for (int u = 0; u < U; u++) s[u] = __ldg(a.aslot + e + u * STREAMS);
      GatherVec<T, VW> y[U];
#pragma unroll
      for (int u = 0; u < U; u++) y[u] = row(s[u]);
#pragma unroll
      for (int u = 0; u < U; u++) add(e + u * STREAMS, y[u]);
    }
    for (; e < e1; e += STREAMS) add(e, row(__ldg(a.aslot + e)));
  }
  // lanes of the same columns, then the warps
#pragma unroll
  for (int o = CL; o < 32; o <<= 1)
#pragma unroll
    for (int l = 0; l < 4; l++)
#pragma unroll
      for (int q = 0; q < VW; q++) acc[l][q] += __shfl_xor_sync(0xffffffffu, acc[l][q], o);
  __shared__ T red[8][4][CL * VW + 1];
  if (lane < CL) {
#pragma unroll
    for (int l = 0; l < 4; l++)
#pragma unroll
      for (int q = 0; q < VW; q++) red[warp][l][cl * VW + q] = acc[l][q];
  }
  __syncthreads();
  for (int o = threadIdx.x; o < 4 * CL * VW; o += 256) {
    const int l = o / (CL * VW), c = o % (CL * VW), v = blockIdx.y * CL * VW + c;
    if (v < a.w) {
      T sum = T(0);
#pragma unroll
      for (int q = 0; q < 8; q++) sum += red[q][l][c];
      a.coef[((int64_t)at * 4 + l) * a.cld + v] = (T)a.energy[4 * at + l] * sum;
    } else if (v < a.zpad) {
      a.coef[((int64_t)at * 4 + l) * a.cld + v] = T(0);
    }
  }
}

// columns covered: w, or zpad when larger
template <typename T, int VW>
cudaError_t launch_gather(const GatherArgs<T>& a, int n_kb, cudaStream_t st) {
  const int cols = std::max(a.w, a.zpad);
  const int64_t wide = (int64_t)n_kb * ((cols + 32 * VW - 1) / (32 * VW));
  if (wide < GATHER_WIDE_CTAS)
    kb_gather_kernel<T, VW, 8><<<dim3(n_kb, (cols + 8 * VW - 1) / (8 * VW)), 256, 0, st>>>(a);
  else
    kb_gather_kernel<T, VW, 32><<<dim3(n_kb, (cols + 32 * VW - 1) / (32 * VW)), 256, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace kscf
