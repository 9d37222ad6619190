// k x k algebra of block sizes 32 and 64, one CTA per block, fp32 throughout: the inverse with everything the steps read from
// it, and the inverse's part of the gradient.  Blocks this small are latency, not work (a 64 x 64 inverse is 0.5 MFLOP), so
// what counts is the number of launches and the length of the chain inside one.  Measured with 28 blocks of 64: Newton-Schulz
// as twelve launches of batched tensor-core products plus splits and the elimination's check about 150 us -> one launch of
// 32 us; 14 blocks of 32 by elimination in global memory 70 us -> 12 us; the gradient's chain (a split and two products, or
// two fp32 products) 22 us -> 7 us.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels_generic.cuh"

namespace cafeq {

// Out = inv(Min) by Gauss-Jordan elimination with partial pivoting, in registers: warp w holds columns [w K/8, (w+1) K/8) of
// every row, lane l the rows l and l + 32.  The warp that owns column p finds the pivot by itself (one integer maximum over
// the bit patterns of the magnitudes) and publishes the column while the others still update theirs; one barrier per step.  Rows are not exchanged: pivot row r_p
// plays row p, and the permutation is applied when the result is written.  Optional: column norms (sum_i Out[i][t]^2), bf16
// hi / lo splits, row-major and transposed.
template <int K>
__global__ void __launch_bounds__(256) small_inverse_kernel(const float* Min, float* __restrict__ Out, float* __restrict__ cnorm,
                                                            uint16_t* __restrict__ hi, uint16_t* __restrict__ lo, uint16_t* __restrict__ thi,
                                                            uint16_t* __restrict__ tlo, int32_t* status) {
  pdl_enter();
  const bool raised = status_raised(status);  // (awaited with the block's loads)
  constexpr int R = K / 32, CW = K / 8;
  __shared__ float tile[K][K + 1];
  __shared__ float fcol[2][K];
  __shared__ int prow[2];
  __shared__ float pinv[2];
  __shared__ int row_of[K], step_of[K];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t base = (size_t)blockIdx.x * K * K;
  for (int e = tid; e < K * K; e += 256) tile[e / K][e % K] = Min[base + e];
  if (__syncthreads_or(raised)) return;
  float a[R][CW];
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int c = 0; c < CW; ++c) a[q][c] = tile[q * 32 + lane][warp * CW + c];
  uint32_t used = 0;  // bit q: row q * 32 + lane has been a pivot
  bool bad = false;
  // the owning warp finds the pivot of column p (register column j) and publishes the column, the pivot's row and reciprocal
  auto publish = [&](int p, const float* col) {
    const int buf = p & 1;
    uint32_t key[R], best = 0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      key[q] = (used >> q & 1u) ? 0u : (__float_as_uint(col[q]) & 0x7FFFFFFFu);
      best = max(best, key[q]);
      fcol[buf][q * 32 + lane] = col[q];
    }
    best = __reduce_max_sync(0xffffffffu, best);
    const bool ok = __uint_as_float(best) > 1e-30f && best < 0x7F800000u;  // (a NaN's pattern exceeds infinity's)
    bool done = false;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const uint32_t m = __ballot_sync(0xffffffffu, key[q] == best);
      if (ok && !done && m && lane == __ffs(m) - 1) {
        const int r = q * 32 + lane;
        pinv[buf] = 1.0f / col[q];
        prow[buf] = r;
        row_of[p] = r;
        step_of[r] = p;
      }
      done = done || m;
    }
    if (!ok && lane == 0) prow[buf] = -1;
  };
  if (warp == 0) {
    float col[R];
#pragma unroll
    for (int q = 0; q < R; ++q) col[q] = a[q][0];
    publish(0, col);
  }
  for (int ow = 0; ow < 8 && !bad; ++ow) {
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      const int p = ow * CW + c, buf = p & 1;
      __syncthreads();  // (a buffer is written again after the next barrier: its readers have passed that one)
      const int r = prow[buf];
      if (r < 0) { bad = true; break; }
      const float d = pinv[buf];
      float f[R];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        f[q] = fcol[buf][q * 32 + lane];
        if (q * 32 + lane == r) used |= 1u << q;
      }
      auto update = [&](int j) {
        const bool own = (warp == ow) && (j == c);
        const float src = (R == 2 && r >= 32) ? a[R - 1][j] : a[0][j];
        const float pv = own ? d : __shfl_sync(0xffffffffu, src, r & 31) * d;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const float x = fmaf(-f[q], pv, own ? 0.f : a[q][j]);
          a[q][j] = (q * 32 + lane == r) ? pv : x;
        }
      };
      // the next column first: its pivot is searched while the other warps update
      constexpr int last = CW - 1;
      const int jn = (c == last) ? 0 : c + 1;
      update(jn);
      if (warp == (c == last ? ow + 1 : ow)) {
        float col[R];
#pragma unroll
        for (int q = 0; q < R; ++q) col[q] = a[q][jn];
        publish(p + 1, col);
      }
#pragma unroll
      for (int j = 0; j < CW; ++j)
        if (j != jn) update(j);
    }
  }
  if (bad) {
    if (tid == 0) raise_status(status, CAFEQ_ERR_SINGULAR);
    return;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int p = step_of[q * 32 + lane];
#pragma unroll
    for (int j = 0; j < CW; ++j) tile[p][row_of[warp * CW + j]] = a[q][j];
  }
  __syncthreads();
  for (int e = tid; e < K * K; e += 256) {
    const float x = tile[e / K][e % K];
    Out[base + e] = x;
    if (hi) {
      const __nv_bfloat16 h = __float2bfloat16_rn(x);
      hi[base + e] = __bfloat16_as_ushort(h);
      lo[base + e] = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(h)));
    }
    if (thi) {
      const float y = tile[e % K][e / K];
      const __nv_bfloat16 h = __float2bfloat16_rn(y);
      thi[base + e] = __bfloat16_as_ushort(h);
      tlo[base + e] = __bfloat16_as_ushort(__float2bfloat16_rn(y - __bfloat162float(h)));
    }
  }
  if (cnorm && tid < K) {
    float s = 0.f;
    for (int i = 0; i < K; ++i) s = fmaf(tile[i][tid], tile[i][tid], s);
    cnorm[(size_t)blockIdx.x * K + tid] = s;
  }
}

// G -= X^T Gx X^T with X = Minv; Gx given, or (null) scale * X[i][t] * A_t with A_t = Agrp[column / g] or A[t] (Eq. 4).  Both
// operands in shared memory, 4 x 4 outputs per thread from 16-byte reads (the pitch of K + 4 spreads eight rows over the
// banks); the intermediate product takes the place of Gx.
template <int K>
__global__ void __launch_bounds__(K * K / 16) small_chain_kernel(const float* X, const float* Gx,
                                                                 const float* A, const float* Agrp, int g,
                                                                 float scale, float* __restrict__ G, const int32_t* status) {
  pdl_enter();
  if (cta_stopped(status)) return;
  constexpr int N = K * K / 16, T = K / 4;
  __shared__ float4 xs4[K][T + 1], gs4[K][T + 1];
  const int tid = threadIdx.x, ti = tid / T, tj = tid % T;
  const size_t base = (size_t)blockIdx.x * K * K;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = tid + u * N, i = e / T, t = (e % T) * 4;
    const float4 x = *reinterpret_cast<const float4*>(X + base + (size_t)e * 4);
    xs4[i][e % T] = x;
    if (Gx) gs4[i][e % T] = *reinterpret_cast<const float4*>(Gx + base + (size_t)e * 4);
    else {
      const long long col = (long long)blockIdx.x * K + t;
      float w[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) w[v] = scale * (Agrp ? Agrp[(col + v) / g] : A[col + v]);
      gs4[i][e % T] = make_float4(w[0] * x.x, w[1] * x.y, w[2] * x.z, w[3] * x.w);
    }
  }
  __syncthreads();
  float acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
#pragma unroll 4
  for (int l = 0; l < K; ++l) {  // T1[i][j] = sum_l X[l][i] Gx[l][j]
    const float4 p = xs4[l][ti], q = gs4[l][tj];
    const float pu[4] = {p.x, p.y, p.z, p.w}, qv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(pu[u], qv[v], acc[u][v]);
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    gs4[4 * ti + u][tj] = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
  }
  __syncthreads();
#pragma unroll 2
  for (int l = 0; l < T; ++l) {  // sum_l T1[i][l] X[j][l], rows i = 4 ti + u, columns j = tj + T v
    float4 p[4], q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { p[u] = gs4[4 * ti + u][l]; q[u] = xs4[tj + T * u][l]; }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v)
        acc[u][v] = fmaf(p[u].x, q[v].x, fmaf(p[u].y, q[v].y, fmaf(p[u].z, q[v].z, fmaf(p[u].w, q[v].w, acc[u][v]))));
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) G[base + (size_t)(4 * ti + u) * K + tj + T * v] -= acc[u][v];
}

}  // namespace cafeq
