// Dense-matrix helpers for the pairwise product term (Eq. 5) and Algorithm 1: bf16 split / transpose of
// rectangular fp32 matrices (the operand layouts of the tensor-core product kernel), replica fold / expansion
// of the inner dimension, and the small control kernels of the iterative pseudo-inverse.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels_gemm.cuh"

namespace cafeq {

// 2^-e with 4^e <= n2 < 4^(e + 1): the power of two that brings a matrix of squared norm n2 to a norm in [1, 2).  Exact as a factor,
// so nothing but the exponents of what is computed from the matrix changes.  (e within the exponents of normal fp32 numbers; a norm
// of zero or one that is not finite takes an end of that range.)
__device__ __forceinline__ double unit_scale(const double n2) {
  const int e = n2 > 0.0 ? (n2 < 1e300 ? ilogb(n2) >> 1 : 126) : 0;
  return ldexp(1.0, -min(max(e, -126), 126));
}

// X fp32 [R, C] (row pitch ld) times `scale` (or times 1 / *inv_scale when inv_scale is given, times unit_scale(*norm2) when norm2
// is) ->
// bf16 hi / lo splits, row-major [R, C] and / or transposed [C, R]; optional fp32 copy Y of the scaled values
// (row-major) and YT (transposed, holding hi + lo: used only as a starting guess).  h3 / t3: optional third term
// bf16(x - hi - lo) in row-major / transposed order (hi + lo + third carries 24 significand bits: products over the
// three-way split reach fp32 accuracy).
// One 64 x 64 tile per CTA (grid: C / 64, R / 64; every caller's sizes are multiples of 64).  Memory-bound: two values per
// thread and access, so that every row of a tile is a 128-byte line in both orders (one value each, 32 x 32 tiles: 22 us for
// the two row-major terms of 3584 x 2048, 9 us here).
__global__ void __launch_bounds__(256) split_rect_kernel(const float* X, int R, int C, long long ld, float scale,
                                                         const double* inv_scale, float* __restrict__ Y,
                                                         float* __restrict__ YT, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo,
                                                         uint16_t* __restrict__ thi, uint16_t* __restrict__ tlo,
                                                         const int32_t* status, uint16_t* __restrict__ h3 = nullptr,
                                                         uint16_t* __restrict__ t3 = nullptr, const double* norm2 = nullptr) {
  pdl_enter();
  if (cta_stopped(status)) return;
  __shared__ uint32_t tile[64][65];
  __shared__ uint16_t tile3[64][66];
  const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float sc = scale;
  if (inv_scale || norm2)
    sc = (float)((double)scale * (norm2 ? unit_scale(*norm2) : 1.0) / (inv_scale ? fmax(*inv_scale, 1e-300) : 1.0));
  const bool trans = thi || tlo || YT;
  float2 x2[8];
  if (((uintptr_t)X & 7) == 0 && (ld & 1) == 0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) x2[q] = ld_plain(reinterpret_cast<const float2*>(X + (long long)(r0 + ty + 8 * q) * ld + c0 + 2 * tx));
  } else {  // (the caller's product may be any float array)
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float* x = X + (long long)(r0 + ty + 8 * q) * ld + c0 + 2 * tx;
      x2[q] = make_float2(x[0], x[1]);
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = ty + 8 * q;
    const long long o = (long long)(r0 + i) * C + c0 + 2 * tx;
    const float x[2] = {sc * x2[q].x, sc * x2[q].y};
    uint32_t hw = 0, lw = 0, w3 = 0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const __nv_bfloat16 h = __float2bfloat16_rn(x[e]);
      const float d = x[e] - __bfloat162float(h);
      const __nv_bfloat16 l = __float2bfloat16_rn(d);
      const uint32_t hb = __bfloat16_as_ushort(h), lb = __bfloat16_as_ushort(l);
      hw |= hb << (16 * e);
      lw |= lb << (16 * e);
      if (trans) tile[i][2 * tx + e] = hb | (lb << 16);
      if (h3 || t3) {
        const uint32_t b3 = __bfloat16_as_ushort(__float2bfloat16_rn(d - __bfloat162float(l)));
        w3 |= b3 << (16 * e);
        tile3[i][2 * tx + e] = (uint16_t)b3;
      }
    }
    if (Y) *reinterpret_cast<float2*>(Y + o) = make_float2(x[0], x[1]);
    if (hi) *reinterpret_cast<uint32_t*>(hi + o) = hw;
    if (lo) *reinterpret_cast<uint32_t*>(lo + o) = lw;
    if (h3) *reinterpret_cast<uint32_t*>(h3 + o) = w3;
  }
  if (!trans && !t3) return;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int j = ty + 8 * q;
    const long long o = (long long)(c0 + j) * R + r0 + 2 * tx;
    if (t3) *reinterpret_cast<uint32_t*>(t3 + o) = (uint32_t)tile3[2 * tx][j] | ((uint32_t)tile3[2 * tx + 1][j] << 16);
    if (trans) {
      const uint32_t v0 = tile[2 * tx][j], v1 = tile[2 * tx + 1][j];
      if (thi) *reinterpret_cast<uint32_t*>(thi + o) = (v0 & 0xFFFFu) | (v1 << 16);
      if (tlo) *reinterpret_cast<uint32_t*>(tlo + o) = (v0 >> 16) | (v1 & 0xFFFF0000u);
      if (YT)
        *reinterpret_cast<float2*>(YT + o) = make_float2(__uint_as_float(v0 << 16) + __uint_as_float(v0 & 0xFFFF0000u),
                                                         __uint_as_float(v1 << 16) + __uint_as_float(v1 & 0xFFFF0000u));
    }
  }
}

// Bf[B*k + j][y] = sum_rep V[y][(B*r + rep)*k + j]: fold the r replicas of every block of the inner dimension
// and transpose (V fp32 [d3, r*h] -> Bf fp32 [h, d3]).  grid: ceil(d3/32), h/32 (k % 32 == 0); block 32 x 8.
__global__ void __launch_bounds__(256) fold_transpose_kernel(const float* V, int d3, int h, int k, int r,
                                                             float* __restrict__ Bf) {
  pdl_enter();
  __shared__ float tile[32][33];
  const int y0 = blockIdx.x * 32, l0 = blockIdx.y * 32;  // l0 inside one block of k
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int B = l0 / k, j0 = l0 - B * k;
  const long long ldv = (long long)r * h;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int y = y0 + ty + 8 * q;
    float s = 0.f;
    if (y < d3)
      for (int rep = 0; rep < r; ++rep) s += V[(long long)y * ldv + (long long)(B * r + rep) * k + j0 + tx];
    tile[ty + 8 * q][tx] = s;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int l = l0 + ty + 8 * q, y = y0 + tx;
    if (y < d3) Bf[(long long)l * d3 + y] = tile[tx][ty + 8 * q];
  }
}

// V[y][(B*r + rep)*k + j] = scale * X[y][B*k + j]  (X fp32 [d3, h] -> V fp32 [d3, r*h]; k % 4 == 0).  grid: (d3,
// ceil(h / 1024)) -- d3 may exceed what the second dimension of a grid holds; a thread reads four entries once and writes every
// replica (60 -> 12 us at 3584 x 4096).
__global__ void __launch_bounds__(256) expand_cols_kernel(const float* X, int h, int k, int r, float scale,
                                                          float* __restrict__ V) {
  pdl_enter();
  const int l = (blockIdx.y * 256 + threadIdx.x) * 4;
  if (l >= h) return;
  const long long y = blockIdx.x;
  float4 x = ld_plain(reinterpret_cast<const float4*>(X + y * h + l));
  x = make_float4(scale * x.x, scale * x.y, scale * x.z, scale * x.w);
  const int B = l / k, j = l - B * k;
  float* v = V + y * (long long)r * h + (long long)B * r * k + j;
  for (int rep = 0; rep < r; ++rep) *reinterpret_cast<float4*>(v + (long long)rep * k) = x;
}

// the same for any k, one entry per thread (learned offsets take every shape)
__global__ void expand_cols_any_kernel(const float* X, int d3, int h, int k, int r, float scale, float* __restrict__ V) {
  pdl_enter();
  const long long n = (long long)d3 * r * h;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const long long y = e / ((long long)r * h);
    const int l = (int)(e - y * (long long)r * h);
    const int Bq = l / k, j = l - Bq * k;
    V[e] = scale * X[y * h + (long long)(Bq / r) * k + j];
  }
}

// bf16 hi / lo (and third) terms of the replica-folded V: F[y][B*k + j] = sum_rep V[y][(B*r + rep)*k + j], row-major [d3, h].
// A product over the r*h expanded inner indices equals the product over the h folded ones: 1 / r of the work.  grid: (d3,
// ceil(h / 1024)).
__global__ void __launch_bounds__(256) fold_split_kernel(const float* V, int h, int k, int r, uint16_t* __restrict__ hi,
                                                         uint16_t* __restrict__ lo, uint16_t* __restrict__ h3, const int32_t* status) {
  pdl_enter();
  if (status && *status) return;
  const int l = (blockIdx.y * 256 + threadIdx.x) * 4;
  if (l >= h) return;
  const long long y = blockIdx.x;
  const int B = l / k, j = l - B * k;
  const float* v = V + y * (long long)r * h + (long long)B * r * k + j;
  float x[4] = {0.f, 0.f, 0.f, 0.f};
  for (int rep = 0; rep < r; ++rep) {
    const float4 q = ld_plain(reinterpret_cast<const float4*>(v + (long long)rep * k));
    x[0] += q.x; x[1] += q.y; x[2] += q.z; x[3] += q.w;
  }
  uint32_t a[2], b[2], c[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    uint32_t aw = 0, bw = 0, cw = 0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float f = x[2 * q + e];
      const __nv_bfloat16 t1 = __float2bfloat16_rn(f);
      const float d1 = f - __bfloat162float(t1);
      const __nv_bfloat16 t2 = __float2bfloat16_rn(d1);
      const __nv_bfloat16 t3 = __float2bfloat16_rn(d1 - __bfloat162float(t2));
      aw |= (uint32_t)__bfloat16_as_ushort(t1) << (16 * e);
      bw |= (uint32_t)__bfloat16_as_ushort(t2) << (16 * e);
      cw |= (uint32_t)__bfloat16_as_ushort(t3) << (16 * e);
    }
    a[q] = aw; b[q] = bw; c[q] = cw;
  }
  const long long o = y * h + l;
  *reinterpret_cast<uint2*>(hi + o) = make_uint2(a[0], a[1]);
  *reinterpret_cast<uint2*>(lo + o) = make_uint2(b[0], b[1]);
  if (h3) *reinterpret_cast<uint2*>(h3 + o) = make_uint2(c[0], c[1]);
}

// gX[row][G*g + idx[row, G]] += coef[row, G]: the scale path of the straight-through quantiser lands on the
// arg-max entry of its group (records row-major)
__global__ void add_argmax_kernel(float* __restrict__ gX, long long ld, int rows, int ng, int g, const float* coef,
                                  const int* idx, const int32_t* status) {
  pdl_enter();
  if (status && *status) return;
  const long long n = (long long)rows * ng;
  for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < n; w += (long long)gridDim.x * blockDim.x) {
    const long long row = w / ng;
    const int G = (int)(w - row * ng);
    gX[row * ld + (long long)G * g + idx[w]] += coef[w];
  }
}

// Gradient with respect to the quantiser's input, ready as an operand: gX (d loss / d Uhat, fp32, pitch ldg) passes through,
// the scale's part sign(U at arg-max) / qmax * sum_e gX_e (q_e - U_e / s) is added at the group's arg-max entry, and the sum is
// written as a bf16 hi / lo split.  U dense [rows, ng g]; r > 1: gX holds one column for the r replicas of each inner column
// (block b of k columns reads block b / r).  Memory-bound, 8 bytes read and 4 written per value: LPG lanes own a group and keep
// it in registers.  3584 x 4096 + 2048 x 3584: expansion, scale path with two divisions per value, arg-max addition and split
// 190 us as seven launches, 60 us here as two.
template <int LPG, int NV>
__global__ void __launch_bounds__(256) ste_grad_split_kernel(const float* U, const float* gX, long long ldg, int rows,
                                                             int ng, int g, int k, int r, const float* a,
                                                             const float* usel, const int* idx, float qmax,
                                                             uint16_t* __restrict__ hi, uint16_t* __restrict__ lo, const int32_t* status) {
  pdl_enter();
  if (warp_stopped(status)) return;
  const int l = threadIdx.x % LPG;
  const long long total = (long long)rows * ng;
  const long long w = (blockIdx.x * 256ll + threadIdx.x) / LPG;
  const bool live = w < total;
  const long long wc = live ? w : total - 1;
  const int row = (int)(wc / ng), G = (int)(wc - (long long)row * ng);
  const long long u0 = (long long)row * ng * g + (long long)G * g;
  const float* gr = gX + (long long)row * ldg;
  float4 u4[NV], d4[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int e = (l + i * LPG) * 4;
    u4[i] = d4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < g) {
      u4[i] = ld_plain(reinterpret_cast<const float4*>(U + u0 + e));
      int col = G * g + e;
      if (r > 1) {
        const int b = col / k;
        col = (b / r) * k + (col - b * k);
      }
      d4[i] = ld_plain(reinterpret_cast<const float4*>(gr + col));
    }
  }
  const float av = a[wc], us = usel[wc];
  const int am = idx[wc];
  const float s = __fdiv_rn(av, qmax);
  const float rs = (s > 0.f) ? __frcp_rn(s) : 0.f;
  const bool fast = rs < 3.0e38f;
  const float win = 0.5f - (qmax + 1.f) * 1.0e-6f;
  constexpr float MAGIC = 12582912.f;
  float sum = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const float u[4] = {u4[i].x, u4[i].y, u4[i].z, u4[i].w}, dv[4] = {d4[i].x, d4[i].y, d4[i].z, d4[i].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // U / s with one correction step; the quotient's rounding as in the quantiser (exact division next to a half-integer)
      const float x0 = u[j] * rs;
      float x = fmaf(fmaf(-s, x0, u[j]), rs, x0);
      float q = (x + MAGIC) - MAGIC;
      if (!(fabsf(x - q) <= win) || !fast) {
        x = (s > 0.f) ? __fdiv_rn(u[j], s) : 0.f;
        q = fminf(fmaxf(rintf(x), -qmax), qmax);
      }
      sum = fmaf(dv[j], q - x, sum);
    }
  }
  for (int o = LPG / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (!live) return;
  const float cf = sum * ((us > 0.f) ? 1.f : ((us < 0.f) ? -1.f : 0.f)) / qmax;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int e = (l + i * LPG) * 4;
    if (e >= g) break;
    const float dv[4] = {d4[i].x, d4[i].y, d4[i].z, d4[i].w};
    uint32_t hw[2] = {0u, 0u}, lw[2] = {0u, 0u};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float x = dv[j] + ((e + j == am) ? cf : 0.f);
      const __nv_bfloat16 h = __float2bfloat16_rn(x);
      hw[j >> 1] |= (uint32_t)__bfloat16_as_ushort(h) << (16 * (j & 1));
      lw[j >> 1] |= (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(h))) << (16 * (j & 1));
    }
    *reinterpret_cast<uint2*>(hi + u0 + e) = make_uint2(hw[0], hw[1]);
    *reinterpret_cast<uint2*>(lo + u0 + e) = make_uint2(lw[0], lw[1]);
  }
}

// Scale path of the straight-through quantiser from the residual itself: with Uhat = s q and Delta = Uhat - U the
// derivative of Uhat with respect to the scale is q - U / s = Delta / s, and s = a / qmax, so the coefficient routed
// to the group's arg-max entry is sign(U at arg-max) / qmax * sum_e gDelta_e Delta_e / s = sign * sum_e gDelta_e Delta_e / a.
// Delta comes as a two-term bf16 split (row pitch ldd); records are group-major when gm is set.  One warp per record.
__global__ void ste_scale_coef_kernel(const float* gD, long long ldg, const uint16_t* Dh,
                                      const uint16_t* Dl, long long ldd, int rows, int ng, int g,
                                      const float* a, const float* usel, int gm,
                                      float* __restrict__ coef, const int32_t* status) {
  pdl_enter();
  if (warp_stopped(status)) return;
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= (long long)rows * ng) return;
  // consecutive warps take consecutive groups of one row (the rows of gD and Delta are read contiguously)
  const int row = (int)(w / ng), G = (int)(w - (long long)row * ng);
  const long long pi = gm ? (long long)G * rows + row : w;
  const float av = a[pi], u = usel[pi];
  const long long c0 = (long long)G * g;
  float sum = 0.f;
  for (int e0 = lane; e0 < g; e0 += 128) {  // (four values requested before the first is used: 33 -> 28 us at 4096 x 3584)
    float x[4], d[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e = e0 + 32 * j;
      x[j] = d[j] = 0.f;
      if (e < g) {
        x[j] = gD[row * ldg + c0 + e];
        d[j] = bf16_bits_to_float(Dh[row * ldd + c0 + e]) + bf16_bits_to_float(Dl[row * ldd + c0 + e]);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) sum = fmaf(x[j], d[j], sum);
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) {
    const float sgn = (u > 0.f) ? 1.f : ((u < 0.f) ? -1.f : 0.f);
    coef[pi] = (av > 0.f) ? sgn * sum / av : 0.f;
  }
}

// acc += sum x[i] y[i]  (fp32 products summed in double; one atomic per block)
__global__ void __launch_bounds__(256) dot_f32_kernel(const float* x, const float* y, long long n,
                                                      double* acc) {
  pdl_enter();
  __shared__ double red[32];
  double s = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    s += (double)(x[e] * y[e]);
  s = block_sum_double(s, red);
  if (threadIdx.x == 0 && s != 0.0) atomicAdd(acc, s);
}

// Start of the Gram iteration: G = A A^T (fp32 [m, m], tiles of 256 on and above the diagonal) -> B0 = G / c with c = 1.0001 ||G||_F,
// so that its eigenvalues lie in [0, 1], and Y1 = (2 mu I - mu^2 B0) / c, both as fp32 (same tiles; B in place of G) and as bf16
// splits of the whole symmetric matrix.  A row of zeros in A sets *singular, and the first residual to one that a start is not used at.
// One 64 x 64 tile per CTA (grid: m / 64, m / 64); memory-bound.
__global__ void __launch_bounds__(256) gram_start_kernel(float* G, int m, const double* fro2, float mu, float* __restrict__ Y,
                                                         uint16_t* __restrict__ Bh, uint16_t* __restrict__ Bl,
                                                         uint16_t* __restrict__ Yh, uint16_t* __restrict__ Yl,
                                                         double* __restrict__ singular, double* __restrict__ first,
                                                         const int32_t* status) {
  pdl_enter();
  if (cta_stopped(status)) return;
  if ((blockIdx.x >> 2) < (blockIdx.y >> 2)) return;
  __shared__ uint32_t tb[64][65], ty[64][65];
  const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
  const int tx = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double c = 1.0001 * sqrt(*fro2);
  const float inv = c > 0.0 ? (float)(1.0 / c) : 0.f;
  auto split = [](float x) -> uint32_t {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    return (uint32_t)__bfloat16_as_ushort(h) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(h))) << 16);
  };
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = w + 8 * q, row = r0 + i, col = c0 + 2 * tx;
    const long long o = (long long)row * m + col;
    const float2 g = ld_plain(reinterpret_cast<const float2*>(G + o));
    if ((row == col && g.x == 0.f) || (row == col + 1 && g.y == 0.f)) { *singular = 1.0; *first = 1e300; }  // (a row of zeros)
    const float2 b = make_float2(g.x * inv, g.y * inv);
    const float2 y = make_float2(((row == col ? 2.f * mu : 0.f) - mu * mu * b.x) * inv, ((row == col + 1 ? 2.f * mu : 0.f) - mu * mu * b.y) * inv);
    *reinterpret_cast<float2*>(G + o) = b;
    *reinterpret_cast<float2*>(Y + o) = y;
    const uint32_t b0 = split(b.x), b1 = split(b.y), y0 = split(y.x), y1 = split(y.y);
    *reinterpret_cast<uint32_t*>(Bh + o) = (b0 & 0xFFFFu) | (b1 << 16);
    *reinterpret_cast<uint32_t*>(Bl + o) = (b0 >> 16) | (b1 & 0xFFFF0000u);
    *reinterpret_cast<uint32_t*>(Yh + o) = (y0 & 0xFFFFu) | (y1 << 16);
    *reinterpret_cast<uint32_t*>(Yl + o) = (y0 >> 16) | (y1 & 0xFFFF0000u);
    tb[i][2 * tx] = b0; tb[i][2 * tx + 1] = b1;
    ty[i][2 * tx] = y0; ty[i][2 * tx + 1] = y1;
  }
  if ((blockIdx.x >> 2) == (blockIdx.y >> 2)) return;  // (diagonal tiles are stored whole)
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int j = w + 8 * q;
    const long long o = (long long)(c0 + j) * m + r0 + 2 * tx;
    const uint32_t b0 = tb[2 * tx][j], b1 = tb[2 * tx + 1][j], y0 = ty[2 * tx][j], y1 = ty[2 * tx + 1][j];
    *reinterpret_cast<uint32_t*>(Bh + o) = (b0 & 0xFFFFu) | (b1 << 16);
    *reinterpret_cast<uint32_t*>(Bl + o) = (b0 >> 16) | (b1 & 0xFFFF0000u);
    *reinterpret_cast<uint32_t*>(Yh + o) = (y0 & 0xFFFFu) | (y1 << 16);
    *reinterpret_cast<uint32_t*>(Yl + o) = (y0 >> 16) | (y1 & 0xFFFF0000u);
  }
}

__global__ void sqrt_hist_kernel(const double* sq, float* __restrict__ out, int n) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (float)sqrt(fmax(sq[i], 0.0));
}

}  // namespace cafeq
