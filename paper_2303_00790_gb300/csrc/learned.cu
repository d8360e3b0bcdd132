// Learned SCF start: radial descriptors of the atoms around every grid point and a
// 32 -> 128 -> 128 -> 1 tanh multilayer perceptron that maps them to a correction of the
// superposition starting potential (the paper has no learned part; this is the
// project's own addition to the SCF start).  Forward, backward (mean squared error) and
// Adam are hand-written kernels; the network is trained on the GPU.
//
// Descriptors: D[p, 16 s + q] = sum over atoms a of species s (s = 0: Si, 1: H) with
// r = |p - R_a| < 8 bohr of exp(-(r - c_q)^2 / (2 sigma^2)) (1 + cos(pi r / 8)) / 2,
// c_q = q * 8/15, sigma = 8/15.
// Network on standardised inputs x = (D - mu) * inv_sd:
//   h1 = tanh(x W1 + b1), h2 = tanh(h1 W2 + b2), y = h2 . w3 + b3.
// Parameter vector (KSCF_MLP_N_PARAMS floats): W1 (32 x 128 row-major), b1, W2 (128 x 128
// row-major), b2, w3, b3.
//
// A block of the MLP kernels takes an equal share of the points in tiles of at most 112 (at
// 16,384 points and 152 blocks one tile of 108 each; tiles of 64 left most blocks a nearly empty
// second one); the weights stay in shared memory for the whole launch.  A thread owns 4 points x
// 8 hidden units of each layer output (points t/16 + 32 r; units 4 (t%16) + c and 64 more, or
// t%16 + 16 c where the weights are walked along their rows) and 8 x 4 weights of dW2.  All
// operands come as 16-byte loads (rows padded by four floats: no bank conflicts), 12 per 128
// multiply-adds instead of 12 scalar ones per 32, and 16 warps share an SM instead of 8: the
// gradient of 16,384 points 91 -> 66 us (29 us at the FP32 rate).  The backward kernel
// keeps its share of the weight gradients in registers across all tiles and writes one partial
// gradient per block; a second kernel adds the partials in FP64 in a fixed order.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "kscf_internal.h"

namespace kscf {
namespace {

constexpr int NIN = KSCF_MLP_N_IN;    // 32
constexpr int NH = KSCF_MLP_N_HID;    // 128
constexpr int NPAR = KSCF_MLP_N_PARAMS;
constexpr int TP = 112;               // most points per tile
constexpr int NT = 512;               // threads per block
constexpr int HS = NH + 4;            // padded row stride of W2 and of the activations
constexpr int XS = NIN + 4;           // padded row stride of the input tile
// parameter offsets
constexpr int OW1 = 0, OB1 = NIN * NH, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH, OB3 = OW3 + NH;
static_assert(OB3 + 1 == NPAR, "parameter layout");

// shared-memory layout (floats)
constexpr int S_W1 = 0;
constexpr int S_W2 = S_W1 + NIN * NH;
constexpr int S_B1 = S_W2 + NH * HS;
constexpr int S_B2 = S_B1 + NH;
constexpr int S_W3 = S_B2 + NH;
constexpr int S_X = S_W3 + NH;
constexpr int S_H1 = S_X + TP * XS;
constexpr int S_H2 = S_H1 + TP * HS;
constexpr int S_Y = S_H2 + TP * HS;      // y, then dy
constexpr int S_T = S_Y + TP;
constexpr int S_ACC = S_T + TP;          // db1, db2, dw3 accumulators of four quarters of a tile (backward)
constexpr int S_END = S_ACC + 12 * NH;
constexpr size_t kMlpSmem = (size_t)S_END * sizeof(float);

__device__ __forceinline__ float to_bf16_value(float x) { return __bfloat162float(__float2bfloat16(x)); }

template <bool BF16>
__device__ __forceinline__ float q(float x) {
  return BF16 ? to_bf16_value(x) : x;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ bool aligned16(const float* p) { return ((uintptr_t)p & 15) == 0; }
template <bool BF16>
__device__ __forceinline__ float4 q4(float4 v) {
  return make_float4(q<BF16>(v.x), q<BF16>(v.y), q<BF16>(v.z), q<BF16>(v.w));
}

// Loads the weights (rounded to bf16 when BF16) into shared memory.
template <bool BF16>
__device__ void load_weights(const float* __restrict__ P, float* sm) {
  if (aligned16(P)) {
    static_assert(OW2 % 4 == 0 && NIN * NH % (4 * NT) == 0 && NH * NH % (4 * NT) == 0, "whole vectors per thread");
    float4 w1[NIN * NH / 4 / NT], w2[NH * NH / 4 / NT];   // all loads before the first store
#pragma unroll
    for (int u = 0; u < NIN * NH / 4 / NT; u++) w1[u] = __ldg((const float4*)(P + OW1) + threadIdx.x + u * NT);
#pragma unroll
    for (int u = 0; u < NH * NH / 4 / NT; u++) w2[u] = __ldg((const float4*)(P + OW2) + threadIdx.x + u * NT);
#pragma unroll
    for (int u = 0; u < NIN * NH / 4 / NT; u++) *(float4*)(sm + S_W1 + 4 * (threadIdx.x + u * NT)) = q4<BF16>(w1[u]);
#pragma unroll
    for (int u = 0; u < NH * NH / 4 / NT; u++) {
      const int e = 4 * (threadIdx.x + u * NT);
      *(float4*)(sm + S_W2 + (e / NH) * HS + e % NH) = q4<BF16>(w2[u]);
    }
  } else {
    for (int e = threadIdx.x; e < NIN * NH; e += NT) sm[S_W1 + e] = q<BF16>(P[OW1 + e]);
    for (int e = threadIdx.x; e < NH * NH; e += NT) sm[S_W2 + (e / NH) * HS + (e % NH)] = q<BF16>(P[OW2 + e]);
  }
  for (int e = threadIdx.x; e < NH; e += NT) {
    sm[S_B1 + e] = P[OB1 + e];
    sm[S_B2 + e] = P[OB2 + e];
    sm[S_W3 + e] = q<BF16>(P[OW3 + e]);
  }
}

// Tiles of at most TP points, or of SMALL where no block has more (n <= 64 per block: up to 9,728
// points): the products run over whole tiles of TE points, so a tile of 112 for 64 points
// wastes 40 % of them (4,000 points: gradient and Adam step 115 -> 97 us).
constexpr int SMALL = 64;
__host__ __device__ constexpr int rows_of(int te) { return (te + 31) / 32; }   // per thread

// Standardised input tile: rows p0 .. p0 + TE - 1 (rows from n on are zero).
template <bool BF16, int TE>
__device__ void load_tile(const float* __restrict__ D, const float* __restrict__ mu, const float* __restrict__ inv_sd,
                          int64_t n, int64_t p0, float* sm) {
  if (aligned16(D) && aligned16(mu) && aligned16(inv_sd)) {
    const int i = 4 * (threadIdx.x % (NIN / 4));   // NT is a multiple of NIN / 4
    const float4 m = __ldg((const float4*)(mu + i)), s = __ldg((const float4*)(inv_sd + i));
#pragma unroll
    for (int e = threadIdx.x; e < TE * NIN / 4; e += NT) {
      const int p = e / (NIN / 4);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (p0 + p < n) {
        v = __ldg((const float4*)(D + (p0 + p) * NIN + i));
        v = make_float4((v.x - m.x) * s.x, (v.y - m.y) * s.y, (v.z - m.z) * s.z, (v.w - m.w) * s.w);
      }
      *(float4*)(sm + S_X + p * XS + i) = q4<BF16>(v);
    }
    return;
  }
  for (int e = threadIdx.x; e < TE * NIN; e += NT) {
    const int p = e / NIN, i = e % NIN;
    const int64_t row = p0 + p;
    float v = 0.0f;
    if (row < n) v = (D[row * NIN + i] - mu[i]) * inv_sd[i];
    sm[S_X + p * XS + i] = q<BF16>(v);
  }
}

template <int TE>
__device__ __forceinline__ int tile_row(int pr, int r) { return min(pr + 32 * r, TE - 1); }

// acc[r][c] += sum_k A[pr + 32 r][k] W[k][col(c)] over k < K, col(c) = 4 hc + c, 64 + 4 hc + c - 4;
// rows past the tile are clamped to its last one and not stored
template <int K, int TE>
__device__ __forceinline__ void layer_product(const float* A, int as, const float* W, int ws, int pr, int hc,
                                              float (&acc)[rows_of(TE)][8]) {
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float4 a4[rows_of(TE)];
#pragma unroll
    for (int r = 0; r < rows_of(TE); r++) a4[r] = ld4(A + tile_row<TE>(pr, r) * as + k);
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const float4 w0 = ld4(W + (k + u) * ws + 4 * hc), w1 = ld4(W + (k + u) * ws + 64 + 4 * hc);
      const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
      for (int r = 0; r < rows_of(TE); r++) {
        const float av = u == 0 ? a4[r].x : u == 1 ? a4[r].y : u == 2 ? a4[r].z : a4[r].w;
#pragma unroll
        for (int c = 0; c < 8; c++) acc[r][c] = fmaf(av, wv[c], acc[r][c]);
      }
    }
  }
}

// h1, h2 and y of the tile in shared memory
template <bool BF16, int TE>
__device__ void forward_tile(float* sm, float b3) {
  const int t = threadIdx.x, pr = t >> 4, hc = t & 15;
  float acc[rows_of(TE)][8];
  auto start = [&](int bias) {
    const float4 b0 = ld4(sm + bias + 4 * hc), b1 = ld4(sm + bias + 64 + 4 * hc);
#pragma unroll
    for (int r = 0; r < rows_of(TE); r++) {
      acc[r][0] = b0.x, acc[r][1] = b0.y, acc[r][2] = b0.z, acc[r][3] = b0.w;
      acc[r][4] = b1.x, acc[r][5] = b1.y, acc[r][6] = b1.z, acc[r][7] = b1.w;
    }
  };
  auto finish = [&](int dst) {
#pragma unroll
    for (int r = 0; r < rows_of(TE); r++)
      if (pr + 32 * r < TE)
#pragma unroll
        for (int h = 0; h < 2; h++)
          *(float4*)(sm + dst + (pr + 32 * r) * HS + 64 * h + 4 * hc) =
              make_float4(q<BF16>(tanhf(acc[r][4 * h])), q<BF16>(tanhf(acc[r][4 * h + 1])),
                          q<BF16>(tanhf(acc[r][4 * h + 2])), q<BF16>(tanhf(acc[r][4 * h + 3])));
  };
  start(S_B1);
  layer_product<NIN, TE>(sm + S_X, XS, sm + S_W1, NH, pr, hc, acc);
  finish(S_H1);
  __syncthreads();
  start(S_B2);
  layer_product<NH, TE>(sm + S_H1, HS, sm + S_W2, HS, pr, hc, acc);
  finish(S_H2);
  __syncthreads();
  // output: warp w handles points w TE / 16 .. + TE / 16 - 1
  const int warp = t >> 5, lane = t & 31;
#pragma unroll
  for (int pp = 0; pp < TE / (NT / 32); pp++) {
    const int p = warp * (TE / (NT / 32)) + pp;
    float s = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; c++) s = fmaf(sm[S_H2 + p * HS + lane + 32 * c], sm[S_W3 + lane + 32 * c], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sm[S_Y + p] = s + b3;
  }
  __syncthreads();
}

template <bool BF16, int TE>
__global__ void __launch_bounds__(NT, 1) mlp_forward_kernel(const float* __restrict__ P, const float* __restrict__ mu,
                                                           const float* __restrict__ inv_sd,
                                                           const float* __restrict__ D, int64_t n,
                                                           float* __restrict__ y) {
  extern __shared__ __align__(16) float sm[];
  load_weights<BF16>(P, sm);
  const float b3 = P[OB3];
  // the block's share of the points
  const int64_t per = (n + gridDim.x - 1) / gridDim.x, r1 = min(n, (blockIdx.x + 1) * per);
  for (int64_t r0 = blockIdx.x * per; r0 < r1; r0 += TE) {
    __syncthreads();
    load_tile<BF16, TE>(D, mu, inv_sd, r1, r0, sm);
    __syncthreads();
    forward_tile<BF16, TE>(sm, b3);
    for (int p = threadIdx.x; p < TE; p += NT)
      if (r0 + p < r1) y[r0 + p] = sm[S_Y + p];
  }
}

// Loss and gradient: every block handles its share of the points and writes part[block * (NPAR + 1) + q] (q < NPAR: gradient, q = NPAR: sum of (y - t)^2).
template <int TE>
__global__ void __launch_bounds__(NT, 1) mlp_grad_kernel(const float* __restrict__ P, const float* __restrict__ mu,
                                                        const float* __restrict__ inv_sd,
                                                        const float* __restrict__ D, const float* __restrict__ tgt,
                                                        int64_t n, float* __restrict__ part) {
  extern __shared__ __align__(16) float sm[];
  load_weights<false>(P, sm);
  const float b3 = P[OB3];
  const int t = threadIdx.x, pr = t >> 4, hc = t & 15;
  for (int e = t; e < 12 * NH; e += NT) sm[S_ACC + e] = 0.0f;
  // dW2 rows 4 wr + a, 64 + 4 wr + a - 4 and columns 4 wc + c; dW1 rows 4 (t / 64) + a and
  // columns 2 (t % 64) + c
  const int wr = t >> 5, wc = t & 31;
  float gW2[8][4], gW1[4][2];
#pragma unroll
  for (int a = 0; a < 8; a++)
#pragma unroll
    for (int c = 0; c < 4; c++) gW2[a][c] = 0.0f;
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int c = 0; c < 2; c++) gW1[a][c] = 0.0f;
  // column sums over the thread's quarter of the tile
  const int sj = t & (NH - 1), s0 = (t >> 7) * (TE / 4);
  float* sacc = sm + S_ACC + (t >> 7) * 3 * NH;
  float loss = 0.0f, gb3 = 0.0f;
  const float scale = 2.0f / (float)n;
  const int64_t per = (n + gridDim.x - 1) / gridDim.x, row1 = min(n, (blockIdx.x + 1) * per);
  for (int64_t row0 = blockIdx.x * per; row0 < row1; row0 += TE) {
    const int np = (int)min((int64_t)TE, row1 - row0);   // points of this tile
    __syncthreads();
    load_tile<false, TE>(D, mu, inv_sd, row1, row0, sm);
    for (int p = t; p < TE; p += NT) sm[S_T + p] = p < np ? tgt[row0 + p] : 0.0f;
    __syncthreads();
    forward_tile<false, TE>(sm, b3);
    // dy = 2 (y - t) / n for the points of the tile, 0 past n
    if (t < TE) {
      const float r = t < np ? sm[S_Y + t] - sm[S_T + t] : 0.0f;
      loss += r * r;
      sm[S_Y + t] = scale * r;
    }
    __syncthreads();
    // dw3[j] += sum_p dy_p h2[p][j]; db3 += sum_p dy_p
    {
      float s = 0.0f;
#pragma unroll 8
      for (int p = s0; p < s0 + TE / 4; p++) s = fmaf(sm[S_Y + p], sm[S_H2 + p * HS + sj], s);
      sacc[2 * NH + sj] += s;
    }
    if (t == 0) {
      float s = 0.0f;
      for (int p = 0; p < TE; p++) s += sm[S_Y + p];
      gb3 += s;
    }
    __syncthreads();
    // g2 = dy w3 (1 - h2^2), in place over h2
    for (int e = t; e < TE * NH / 4; e += NT) {
      const int p = e >> 5, j = 4 * (e & 31);
      float4 h = ld4(sm + S_H2 + p * HS + j);
      const float4 w = ld4(sm + S_W3 + j);
      const float dy = sm[S_Y + p];
      h.x = dy * w.x * (1.0f - h.x * h.x);
      h.y = dy * w.y * (1.0f - h.y * h.y);
      h.z = dy * w.z * (1.0f - h.z * h.z);
      h.w = dy * w.w * (1.0f - h.w * h.w);
      *(float4*)(sm + S_H2 + p * HS + j) = h;
    }
    __syncthreads();
    // db2[j] += sum_p g2[p][j]; dW2[i][j] += sum_p h1[p][i] g2[p][j]
    {
      float s = 0.0f;
#pragma unroll 8
      for (int p = s0; p < s0 + TE / 4; p++) s += sm[S_H2 + p * HS + sj];
      sacc[NH + sj] += s;
    }
#pragma unroll 2
    for (int p = 0; p < np; p++) {   // (dy, and so g2, is zero from np on)
      const float4 h0 = ld4(sm + S_H1 + p * HS + 4 * wr), h1 = ld4(sm + S_H1 + p * HS + 64 + 4 * wr);
      const float4 g = ld4(sm + S_H2 + p * HS + 4 * wc);
      const float hv[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w}, gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
      for (int a = 0; a < 8; a++)
#pragma unroll
        for (int c = 0; c < 4; c++) gW2[a][c] = fmaf(hv[a], gv[c], gW2[a][c]);
    }
    __syncthreads();
    // g1[p][i] = (sum_j g2[p][j] W2[i][j]) (1 - h1[p][i]^2), in place over h1; units hc + 16 c
    {
      float acc[rows_of(TE)][8];
#pragma unroll
      for (int r = 0; r < rows_of(TE); r++)
#pragma unroll
        for (int c = 0; c < 8; c++) acc[r][c] = 0.0f;
#pragma unroll 2
      for (int j = 0; j < NH; j += 4) {
        float4 g4[rows_of(TE)];
#pragma unroll
        for (int r = 0; r < rows_of(TE); r++) g4[r] = ld4(sm + S_H2 + tile_row<TE>(pr, r) * HS + j);
#pragma unroll
        for (int c = 0; c < 8; c++) {
          const float4 w = ld4(sm + S_W2 + (hc + 16 * c) * HS + j);
#pragma unroll
          for (int r = 0; r < rows_of(TE); r++)
            acc[r][c] = fmaf(g4[r].w, w.w, fmaf(g4[r].z, w.z, fmaf(g4[r].y, w.y, fmaf(g4[r].x, w.x, acc[r][c]))));
        }
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < rows_of(TE); r++)
#pragma unroll
        for (int c = 0; c < 8; c++) {
          const int p = pr + 32 * r, i = hc + 16 * c;
          if (p >= TE) continue;
          const float h = sm[S_H1 + p * HS + i];
          sm[S_H1 + p * HS + i] = acc[r][c] * (1.0f - h * h);
        }
    }
    __syncthreads();
    // db1[i] += sum_p g1[p][i]; dW1[i][j] += sum_p x[p][i] g1[p][j]
    {
      float s = 0.0f;
#pragma unroll 8
      for (int p = s0; p < s0 + TE / 4; p++) s += sm[S_H1 + p * HS + sj];
      sacc[sj] += s;
    }
#pragma unroll 4
    for (int p = 0; p < np; p++) {
      const float4 x = ld4(sm + S_X + p * XS + 4 * (t >> 6));
      const float2 g = *(const float2*)(sm + S_H1 + p * HS + 2 * (t & 63));
      const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int a = 0; a < 4; a++) {
        gW1[a][0] = fmaf(xv[a], g.x, gW1[a][0]);
        gW1[a][1] = fmaf(xv[a], g.y, gW1[a][1]);
      }
    }
  }
  __syncthreads();
  // block partials
  float* out = part + (int64_t)blockIdx.x * (NPAR + 1);
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int c = 0; c < 2; c++) out[OW1 + (4 * (t >> 6) + a) * NH + 2 * (t & 63) + c] = gW1[a][c];
#pragma unroll
  for (int a = 0; a < 8; a++)
#pragma unroll
    for (int c = 0; c < 4; c++) out[OW2 + (4 * wr + (a & 3) + 64 * (a >> 2)) * NH + 4 * wc + c] = gW2[a][c];
  if (t < NH) {
    auto quarters = [&](int o) {
      return (sm[S_ACC + o + t] + sm[S_ACC + 3 * NH + o + t]) + (sm[S_ACC + 6 * NH + o + t] + sm[S_ACC + 9 * NH + o + t]);
    };
    out[OB1 + t] = quarters(0);
    out[OB2 + t] = quarters(NH);
    out[OW3 + t] = quarters(2 * NH);
  }
  if (t == 0) out[OB3] = gb3;
  // loss: threads < TE hold their points' squared residuals
  __shared__ float sl[NT / 32];
  float l = loss;
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((t & 31) == 0) sl[t >> 5] = l;
  __syncthreads();
  if (t == 0) {
    float s = 0.0f;
    for (int w = 0; w < NT / 32; w++) s += sl[w];
    out[NPAR] = s;
  }
}

// Sum of RB floats as an FP64 number, formed in integers: the values are aligned
// to the largest exponent with 57 bits (cut below 2^-57 of the largest, where FP64 additions
// round at 2^-53) and one conversion rounds the sum.  NaN and Inf are added in FP64.
constexpr int RB = 20;
__device__ __forceinline__ double sum_floats(const float (&f)[RB]) {
  int em = 1;
#pragma unroll
  for (int u = 0; u < RB; u++) em = max(em, (__float_as_int(f[u]) >> 23) & 255);
  if (em == 255) {
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < RB; u++) s += (double)f[u];
    return s;
  }
  long long m = 0;
#pragma unroll
  for (int u = 0; u < RB; u++) {
    const int b = __float_as_int(f[u]), e = (b >> 23) & 255;
    const long long x = ((long long)((b & 0x7fffff) | (e ? 0x800000 : 0)) << 33) >> min(em - max(e, 1), 63);
    m += b < 0 ? -x : x;
  }
  return (double)m * __hiloint2double((em - 127 - 23 - 33 + 1023) << 20, 0);
}

// grad[q] = sum_b part[b][q] (FP64, fixed order); loss = sum_b part[b][NPAR] / n.  A block adds 32
// values, each in eight chains of rows that meet in shared memory.  A chain's loads are in
// flight together and its sum is formed in integers: the 152 FP64 additions per value alone took
// 5 us of the FP64 pipe (one chain on 82 blocks 27 us, eight chains 17 us, this 7.4 us with cold
// caches, 12.7 MB of partials).
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float* __restrict__ part, int nb, int64_t n,
                                                         float* __restrict__ grad, double* __restrict__ loss) {
  __shared__ double red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (q <= NPAR) {
    for (int b0 = w; b0 < nb; b0 += 8 * RB) {
      float f[RB];
#pragma unroll
      for (int u = 0; u < RB; u++) {
        const int b = b0 + 8 * u;
        f[u] = b < nb ? __ldg(part + (int64_t)b * (NPAR + 1) + q) : 0.0f;
      }
      const double t = sum_floats(f);
      s = b0 == w ? t : s + t;
    }
  }
  red[w][lane] = s;
  __syncthreads();
  if (w != 0 || q > NPAR) return;
#pragma unroll
  for (int u = 1; u < 8; u++) s += red[u][lane];
  if (q < NPAR)
    grad[q] = (float)s;
  else if (loss)
    loss[0] = s / (double)n;
}

// Adam (Kingma & Ba 2015), step t >= 1
__global__ void adam_kernel(float* __restrict__ P, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Descriptors: one thread per slot; atoms staged through shared memory.
// atoms: 4 floats each (x, y, z relative to the grid centre, species 0/1).
__global__ void descriptor_kernel(const double* __restrict__ rel, const uint8_t* __restrict__ mask,
                                  const float4* __restrict__ atoms, int n_atoms, int64_t n, float* __restrict__ D) {
  __shared__ float4 sa[256];
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = s < n && mask[s];
  float px = 0.f, py = 0.f, pz = 0.f;
  if (live) {
    px = (float)rel[3 * s];
    py = (float)rel[3 * s + 1];
    pz = (float)rel[3 * s + 2];
  }
  float acc[NIN];
#pragma unroll
  for (int j = 0; j < NIN; j++) acc[j] = 0.0f;
  const float rc = KSCF_MLP_R_CUT;
  const float dc = rc / (KSCF_MLP_N_RADIAL - 1);
  const float inv2s2 = 1.0f / (2.0f * dc * dc);
  for (int a0 = 0; a0 < n_atoms; a0 += 256) {
    const int na = min(256, n_atoms - a0);
    __syncthreads();
    if (threadIdx.x < na) sa[threadIdx.x] = atoms[a0 + threadIdx.x];
    __syncthreads();
    if (!live) continue;
    for (int a = 0; a < na; a++) {
      const float4 at = sa[a];
      const float dx = px - at.x, dy = py - at.y, dz = pz - at.z;
      const float r2 = dx * dx + dy * dy + dz * dz;
      if (!(r2 < rc * rc)) continue;
      const float r = sqrtf(r2);
      const float fc = 0.5f * (1.0f + cospif(r / rc));
      const float w_si = at.w == 0.0f ? fc : 0.0f;
      const float w_h = at.w == 0.0f ? 0.0f : fc;
#pragma unroll
      for (int qq = 0; qq < KSCF_MLP_N_RADIAL; qq++) {
        const float d = r - qq * dc;
        const float g = expf(-d * d * inv2s2);
        acc[qq] = fmaf(g, w_si, acc[qq]);
        acc[KSCF_MLP_N_RADIAL + qq] = fmaf(g, w_h, acc[KSCF_MLP_N_RADIAL + qq]);
      }
    }
  }
  if (s < n) {
#pragma unroll
    for (int j = 0; j < NIN; j++) D[s * NIN + j] = acc[j];
  }
}

unsigned mlp_grid(int64_t n) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 63) / 64, sms));   // at least 64 points each
}

// no block of nb has more than SMALL points
bool small_tiles(int64_t n, unsigned nb) { return (n + nb - 1) / nb <= SMALL; }

cudaError_t set_smem_attrs() {
  static bool done = false;
  if (done) return cudaSuccess;
  const void* ks[] = {(const void*)mlp_forward_kernel<false, TP>, (const void*)mlp_forward_kernel<false, SMALL>,
                      (const void*)mlp_forward_kernel<true, TP>,  (const void*)mlp_forward_kernel<true, SMALL>,
                      (const void*)mlp_grad_kernel<TP>,           (const void*)mlp_grad_kernel<SMALL>};
  cudaError_t e = cudaSuccess;
  for (const void* k : ks)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem);
  if (e == cudaSuccess) done = true;
  return e;
}


// ---- standardisation statistics: deterministic FP64 sums over kStdBlocks row ranges ----
constexpr int kStdBlocks = 256, kStdCols = NIN + 1;   // 32 descriptor columns + the target

// part[b][j] = sum over the rows of block b of (x_j - centre_j)^pw (pw = 1 or 2; column NIN
// is the target t); centre null means 0.  Thread (j = tid % 32, g = tid / 32) takes rows
// g, g + 8, ... of the block's range so that one warp reads whole rows.
__global__ void __launch_bounds__(256) std_partial_kernel(const float* __restrict__ D, const float* __restrict__ t,
                                                          int64_t n, const double* __restrict__ centre, int pw,
                                                          double* __restrict__ part) {
  const int j = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t per = (n + kStdBlocks - 1) / kStdBlocks;
  const int64_t r0 = (int64_t)blockIdx.x * per, r1 = min(n, r0 + per);
  const double cj = centre ? centre[j] : 0.0, ct = centre ? centre[NIN] : 0.0;
  double sx = 0.0, st = 0.0;
  for (int64_t r = r0 + g; r < r1; r += 8) {
    const double x = (double)D[r * NIN + j] - cj;
    sx += pw == 1 ? x : x * x;
    if (j == 0) {
      const double y = (double)t[r] - ct;
      st += pw == 1 ? y : y * y;
    }
  }
  __shared__ double red[8][kStdCols];
  red[g][j] = sx;
  if (j == 0) red[g][NIN] = st;
  __syncthreads();
  if (threadIdx.x < kStdCols) {
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < 8; q++) acc += red[q][threadIdx.x];
    part[(int64_t)blockIdx.x * kStdCols + threadIdx.x] = acc;
  }
}

// out[j] = (sum_b part[b][j]) / div in block order
__global__ void std_finish_kernel(const double* __restrict__ part, double div, double* __restrict__ out) {
  const int j = threadIdx.x;
  if (j >= kStdCols) return;
  double acc = 0.0;
  for (int b = 0; b < kStdBlocks; b++) acc += part[(int64_t)b * kStdCols + j];
  out[j] = acc / div;
}

// mu, inv_sd (floor 1e-6), t_shift / t_scale (1 for a constant target) from mean and variance
__global__ void std_params_kernel(const double* __restrict__ mean, const double* __restrict__ var, float* __restrict__ mu,
                                  float* __restrict__ inv_sd, double* __restrict__ shift_scale) {
  const int j = threadIdx.x;
  if (j < NIN) {
    const double sd = sqrt(var[j]);
    mu[j] = (float)mean[j];
    inv_sd[j] = sd > 1e-6 ? (float)(1.0 / sd) : 0.0f;
  } else if (j == NIN) {
    const double sc = sqrt(var[NIN]);
    shift_scale[0] = mean[NIN];
    shift_scale[1] = sc > 0.0 ? sc : 1.0;
  }
}

__global__ void std_target_kernel(const float* __restrict__ t, int64_t n, const double* __restrict__ shift_scale,
                                  float* __restrict__ t_norm) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) t_norm[r] = (float)(((double)t[r] - shift_scale[0]) / shift_scale[1]);
}

__global__ void affine_kernel(const float* __restrict__ y, int64_t n, double scale, double shift,
                              double* __restrict__ dv) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) dv[r] = (double)y[r] * scale + shift;
}
}  // namespace
}  // namespace kscf

using namespace kscf;

extern "C" int kscf_descriptors(const kscf_ham* ham, const kscf_atom* atoms, int n_atoms, float* D, void* stream) {
  if (!ham || !D || n_atoms < 0 || (n_atoms > 0 && !atoms)) {
    set_error("kscf_descriptors: invalid argument");
    return KSCF_ERR_INVALID;
  }
  const Grid& g = ham->h.grid;
  std::vector<float> at(4 * (size_t)std::max(n_atoms, 1));
  for (int a = 0; a < n_atoms; a++) {
    if (atoms[a].z_number != 14 && atoms[a].z_number != 1) {
      set_error("kscf_descriptors: atom %d has Z=%d; descriptors are defined for Si and H", a, atoms[a].z_number);
      return KSCF_ERR_INVALID;
    }
    at[4 * a + 0] = (float)(atoms[a].x - g.center[0]);
    at[4 * a + 1] = (float)(atoms[a].y - g.center[1]);
    at[4 * a + 2] = (float)(atoms[a].z - g.center[2]);
    at[4 * a + 3] = atoms[a].z_number == 14 ? 0.0f : 1.0f;
  }
  std::vector<double> rel(3 * (size_t)g.n_slots);
  for (int64_t s = 0; s < g.n_slots; s++) {
    int ijk[3];
    g.slot_ijk(s, ijk);
    for (int d = 0; d < 3; d++) rel[3 * s + d] = g.h * (double)ijk[d];
  }
  float4* d_at = nullptr;
  double* d_rel = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaMalloc((void**)&d_at, at.size() * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc((void**)&d_rel, rel.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_at, at.data(), at.size() * sizeof(float), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_rel, rel.data(), rel.size() * sizeof(double), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    descriptor_kernel<<<(unsigned)((g.n_slots + 127) / 128), 128, 0, st>>>(d_rel, ham->h.d_mask, d_at, n_atoms,
                                                                          g.n_slots, D);
    count_launch();
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // the host arrays go out of scope
  if (d_at) cudaFree(d_at);
  if (d_rel) cudaFree(d_rel);
  if (e != cudaSuccess) {
    set_error("kscf_descriptors: %s", cudaGetErrorString(e));
    return KSCF_ERR_CUDA;
  }
  return KSCF_OK;
}

extern "C" int kscf_mlp_forward(const float* params, const float* mu, const float* inv_sd, const float* D, int64_t n,
                                int precision, float* y, void* stream) {
  if (!params || !mu || !inv_sd || (n > 0 && (!D || !y)) || n < 0 ||
      (precision != KSCF_MLP_FP32 && precision != KSCF_MLP_BF16)) {
    set_error("kscf_mlp_forward: invalid argument");
    return KSCF_ERR_INVALID;
  }
  if (n == 0) return KSCF_OK;
  KSCF_CUDA_TRY(set_smem_attrs());
  cudaStream_t st = (cudaStream_t)stream;
  const unsigned nb = mlp_grid(n);
  const bool small = small_tiles(n, nb);
  auto k = precision == KSCF_MLP_FP32 ? (small ? mlp_forward_kernel<false, SMALL> : mlp_forward_kernel<false, TP>)
                                      : (small ? mlp_forward_kernel<true, SMALL> : mlp_forward_kernel<true, TP>);
  k<<<nb, NT, kMlpSmem, st>>>(params, mu, inv_sd, D, n, y);
  count_launch();
  KSCF_CUDA_TRY(cudaGetLastError());
  return KSCF_OK;
}

extern "C" int kscf_mlp_work_size(int64_t n, size_t* bytes) {
  if (!bytes || n < 1) {
    set_error("kscf_mlp_work_size: invalid argument");
    return KSCF_ERR_INVALID;
  }
  *bytes = (size_t)mlp_grid(n) * (NPAR + 1) * sizeof(float);
  return KSCF_OK;
}

extern "C" int kscf_mlp_loss_grad(const float* params, const float* mu, const float* inv_sd, const float* D,
                                  const float* t, int64_t n, float* grad, double* loss, void* work, size_t work_bytes,
                                  void* stream) {
  if (!params || !mu || !inv_sd || !D || !t || !grad || n < 1) {
    set_error("kscf_mlp_loss_grad: invalid argument");
    return KSCF_ERR_INVALID;
  }
  const unsigned nb = mlp_grid(n);
  const size_t need = (size_t)nb * (NPAR + 1) * sizeof(float);
  if (!work || work_bytes < need) {
    set_error("kscf_mlp_loss_grad: work buffer of %zu bytes, need %zu", work_bytes, need);
    return KSCF_ERR_WORKSPACE;
  }
  KSCF_CUDA_TRY(set_smem_attrs());
  cudaStream_t st = (cudaStream_t)stream;
  auto k = small_tiles(n, nb) ? mlp_grad_kernel<SMALL> : mlp_grad_kernel<TP>;
  k<<<nb, NT, kMlpSmem, st>>>(params, mu, inv_sd, D, t, n, (float*)work);
  count_launch();
  KSCF_CUDA_TRY(cudaGetLastError());
  mlp_reduce_kernel<<<(NPAR + 1 + 31) / 32, 256, 0, st>>>((const float*)work, (int)nb, n, grad, loss);
  count_launch();
  KSCF_CUDA_TRY(cudaGetLastError());
  return KSCF_OK;
}

extern "C" int kscf_mlp_adam(float* params, const float* grad, float* m, float* v, int step, float lr, float beta1,
                             float beta2, float eps, void* stream) {
  if (!params || !grad || !m || !v || step < 1 || !(lr > 0.0f)) {
    set_error("kscf_mlp_adam: invalid argument");
    return KSCF_ERR_INVALID;
  }
  const float c1 = (float)(1.0 - std::pow((double)beta1, step));
  const float c2 = (float)(1.0 - std::pow((double)beta2, step));
  adam_kernel<<<(NPAR + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, grad, m, v, NPAR, lr, beta1, beta2, eps,
                                                                    c1, c2);
  count_launch();
  KSCF_CUDA_TRY(cudaGetLastError());
  return KSCF_OK;
}

extern "C" int kscf_mlp_standardize(const float* D, const float* t, int64_t n, float* mu, float* inv_sd, float* t_norm,
                                    double* t_shift_scale, void* stream) {
  if (!D || !t || !mu || !inv_sd || !t_norm || !t_shift_scale || n < 2) {
    set_error("kscf_mlp_standardize: invalid argument (n >= 2 rows needed)");
    return KSCF_ERR_INVALID;
  }
  cudaStream_t st = (cudaStream_t)stream;
  double* buf = nullptr;   // partials, mean, variance, shift/scale
  const size_t nbuf = (size_t)kStdBlocks * kStdCols + 3 * kStdCols;
  KSCF_CUDA_TRY(cudaMalloc((void**)&buf, nbuf * sizeof(double)));
  double* part = buf;
  double* mean = part + (size_t)kStdBlocks * kStdCols;
  double* var = mean + kStdCols;
  double* ss = var + kStdCols;
  std_partial_kernel<<<kStdBlocks, 256, 0, st>>>(D, t, n, nullptr, 1, part), count_launch();
  std_finish_kernel<<<1, 64, 0, st>>>(part, (double)n, mean), count_launch();
  std_partial_kernel<<<kStdBlocks, 256, 0, st>>>(D, t, n, mean, 2, part), count_launch();
  std_finish_kernel<<<1, 64, 0, st>>>(part, (double)(n - 1), var), count_launch();
  std_params_kernel<<<1, 64, 0, st>>>(mean, var, mu, inv_sd, ss), count_launch();
  std_target_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(t, n, ss, t_norm), count_launch();
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(t_shift_scale, ss, 2 * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(buf);
  if (e != cudaSuccess) {
    set_error("kscf_mlp_standardize: %s", cudaGetErrorString(e));
    return KSCF_ERR_CUDA;
  }
  return KSCF_OK;
}

extern "C" int kscf_mlp_correction(const float* params, const float* mu, const float* inv_sd, double t_shift,
                                   double t_scale, const float* D, int64_t n, int precision, float* y_work, double* dv,
                                   void* stream) {
  if (!dv || (n > 0 && !y_work) || !std::isfinite(t_shift) || !std::isfinite(t_scale)) {
    set_error("kscf_mlp_correction: invalid argument");
    return KSCF_ERR_INVALID;
  }
  int rc = kscf_mlp_forward(params, mu, inv_sd, D, n, precision, y_work, stream);
  if (rc) return rc;
  if (n == 0) return KSCF_OK;
  affine_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(y_work, n, t_scale, t_shift, dv);
  count_launch();
  KSCF_CUDA_TRY(cudaGetLastError());
  return KSCF_OK;
}
