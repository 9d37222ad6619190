// Fused chains of k x k products on the tensor cores (k = 128 or 256): one CTA carries one operator block through a
// whole chain, so that intermediate results stay in shared memory and no launch separates the products.
#pragma once

#include "kernels_gemm.cuh"

namespace cafeq {

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// all bulk stores of this thread are complete (visible in global memory)
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ------------------------------------------------------------------------------------------------
// Block inverse by Newton-Schulz: X <- X + X (I - A X), as many rounds as the block needs, in one launch.
//   round: R = I - A X over X = hi + lo (two terms, 24-bit products against bf16 A), ||R||_F in the same epilogue,
//          X += hi R (one term: the round corrects its own error), new hi / lo splits, fp32 X on the last round.
// The last round is the one whose residual before the update is below the gate; a block that never gets there is inverted by
// elimination at the end.  The column square norms of the result (Eq. 4's weights) come out of the last update's epilogue.
//
// What bounds it: one round at k = 256 moves 512 KB into the SM (A, hi, lo, hi again) at the 60 - 75 GB/s one SM takes
// from L2, and spends 3 x 1.1 us per 64-column chunk of products; as two launches per round (residual, update) each
// launch paid about 8 us of prologue, pipeline fill and drain on top, and the residual went to memory and back.
// Measured (106 blocks of 256, a step that takes two rounds): 55 us; as separate launches 8 x 17.6 us (the later ones
// gated off).  72 blocks of 128: 17.5 us against 8 x 7.1.  A cold start of 14 blocks of 256: 86 us against 12 x 18.
// R stays in shared memory: written row-major in the 128-byte-swizzled layout of the operand boxes, which the second
// product reads as its MN-major operand.  The updates are in place (a tile is read and written by the same warp after
// every product of the round has read its operands).
// Shared memory: NRING slots + the R area (K / 64 slots); the residual products stream through all slots, the update
// products through the ring, the epilogue's tiles take over both afterwards.
// ------------------------------------------------------------------------------------------------
struct NsMaps {
  CUtensorMap a;       // bf16 A, boxes of K rows x 64 (K-major operand)
  CUtensorMap xh_mn, xl_mn;  // hi / lo of X, boxes of 64 x 64 (MN-major operand)
  CUtensorMap xh_k;    // hi of X, boxes of K rows x 64 (K-major operand)
  CUtensorMap xhl;     // hi and lo as two planes, boxes of 32 x 32 x 2, 64-byte swizzle
  CUtensorMap x;       // fp32 X, boxes of 32 x 32, 128-byte swizzle
};
constexpr int KK_MAX_PROBS = 8;
struct NsParams {
  int max_rounds;
  double gate2;        // squared residual below which a round is the last one
  double accept2;      // a block whose last residual before an update is above this (squared) is inverted by elimination
  const uint16_t* A;   // [nb, K, K]
  uint16_t *hi, *lo;   // splits of X
  float* X;
  int* redo_count;     // optional: blocks inverted by elimination, added up
  // Eq. 4's weights for the blocks of the first n problems (blk0[p] <= b < blk0[p + 1]):
  float* c;            // column square norms c[b][t] = sum_i X[i][t]^2 (may be null)
  int n;
  int blk0[KK_MAX_PROBS + 1];
  float* cw[KK_MAX_PROBS];  // sums of c over runs of g columns of the problem, added to cw (null: none)
  int g[KK_MAX_PROBS];
  int n_ticks;
  float* tick[KK_MAX_PROBS];  // optimiser step counters, advanced by one
  int32_t* status;
};

template <int K>
struct NsCfg {
  static constexpr int HALVES = K / 128;
  static constexpr int KCH = K / 64;
  static constexpr int SLOT = K * 128;
  static constexpr int NRING = (K == 256) ? 3 : 10;
  static constexpr int NSLOT = NRING + KCH;
  static constexpr int EPI_WARPS = 16;
  static constexpr int EPI_WARP_BYTES = 12288;  // two hi + lo tiles (in and out), one fp32 tile
  static constexpr int NBAR = 2 * NSLOT + 3 + 2 * EPI_WARPS;
  static constexpr int SMEM = 1024 + NSLOT * SLOT + 8 * NBAR + 8 * EPI_WARPS + 64 + 4 * K;
  static constexpr int TMEM_COLS = HALVES * K;
  static constexpr int THREADS = 64 + 32 * EPI_WARPS;
  static_assert(NSLOT * SLOT >= EPI_WARPS * EPI_WARP_BYTES, "epilogue tiles must fit");
};

template <int K>
__global__ void __launch_bounds__(NsCfg<K>::THREADS, 1)
ns_block_kernel(const __grid_constant__ NsMaps maps, const __grid_constant__ NsParams p) {
  pdl_wait();  // (releases at its end: a layer's penalty chain shares the SMs with it, which waiting CTAs of the pass would take)
  using C = NsCfg<K>;
  const bool raised = status_raised(p.status);  // (awaited at the end of the set-up)
  const int b = blockIdx.x, row_b = b * K;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + C::NSLOT * C::SLOT);
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8 * C::NSLOT;
  const uint32_t bar_acc = bar_empty + 8 * C::NSLOT;  // a product chain is complete
  const uint32_t bar_r = bar_acc + 8;                 // R and the partial norms are in shared memory
  const uint32_t bar_x = bar_r + 8;                   // the updated X is in global memory
  const uint32_t bar_c0 = bar_x + 8;                  // two per epilogue warp
  double* red = (double*)(bars + C::NBAR);            // [EPI_WARPS] partial squared norms
  uint32_t* tmem_slot = (uint32_t*)(red + C::EPI_WARPS);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sm_u = smem_u32(smem);
  const uint32_t sR = sm_u + C::NRING * C::SLOT;
  volatile int* not_converged = (volatile int*)(tmem_slot + 2);
  float* cn = (float*)(tmem_slot + 16);  // [K] column square norms of the result
  int prob = -1;
  for (int q = 0; q < p.n; ++q)
    if (b >= p.blk0[q] && b < p.blk0[q + 1]) prob = q;
  const bool want_c = prob >= 0 && p.c;
  for (int e = threadIdx.x; e < K; e += C::THREADS) cn[e] = 0.f;

  if (threadIdx.x == 0) {
    *not_converged = 0;
    tma_prefetch_desc(&maps.a);
    tma_prefetch_desc(&maps.xh_mn);
    tma_prefetch_desc(&maps.xl_mn);
    tma_prefetch_desc(&maps.xh_k);
    for (int s = 0; s < C::NSLOT; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    mbar_init(bar_acc, 1);
    mbar_init(bar_r, C::EPI_WARPS);
    mbar_init(bar_x, C::EPI_WARPS);
    for (int s = 0; s < 2 * C::EPI_WARPS; ++s) mbar_init(bar_c0 + 8 * s, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)C::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  const bool stopped = __syncthreads_or(raised) != 0;
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (stopped) {
    if (warp == 1) tmem_free(tmem_base, C::TMEM_COLS);
    return;
  }
  if (b == 0 && threadIdx.x < p.n_ticks && p.tick[threadIdx.x]) *p.tick[threadIdx.x] += 1.f;

  // every role takes the same decision from the same 16 partial sums
  auto residual2 = [&]() {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < C::EPI_WARPS; ++w) s += ((volatile double*)red)[w];
    return s;
  };

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      uint32_t eph = 0xFFFFFFFFu;  // parity of the next wait on each slot's empty barrier (fresh barriers: 1 passes at once)
      bool ok = true;
      for (int it = 0; it < p.max_rounds && ok; ++it) {
        if (it > 0) {
          if (!mbar_wait(bar_x, (it - 1) & 1u, abort_flag, p.status)) break;
          asm volatile("fence.proxy.async;" ::: "memory");
        }
        int s = 0;
        for (int c = 0; c < C::KCH && ok; ++c)
          for (int u = 0; u < 3; ++u) {
            if (!mbar_wait(bar_empty + 8 * s, (eph >> s) & 1u, abort_flag, p.status)) { ok = false; break; }
            eph ^= 1u << s;
            mbar_expect_tx(bar_full + 8 * s, C::SLOT);
            const uint32_t dst = sm_u + s * C::SLOT;
            if (u == 0) {
              tma_load_2d(dst, &maps.a, c * 64, row_b, bar_full + 8 * s);
            } else {
              const CUtensorMap* m = (u == 1) ? &maps.xh_mn : &maps.xl_mn;
              for (int j = 0; j < K / 64; ++j) tma_load_2d(dst + j * 8192, m, j * 64, row_b + c * 64, bar_full + 8 * s);
            }
            if (++s == C::NSLOT) s = 0;
          }
        for (int c = 0; c < C::KCH && ok; ++c) {
          const int sl = c % C::NRING;
          if (!mbar_wait(bar_empty + 8 * sl, (eph >> sl) & 1u, abort_flag, p.status)) { ok = false; break; }
          eph ^= 1u << sl;
          mbar_expect_tx(bar_full + 8 * sl, C::SLOT);
          tma_load_2d(sm_u + sl * C::SLOT, &maps.xh_k, c * 64, row_b, bar_full + 8 * sl);
        }
        if (!ok || !mbar_wait(bar_r, it & 1u, abort_flag, p.status)) break;
        if (residual2() <= p.gate2) break;
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (converged warp, one elected lane)
    constexpr uint32_t idesc = umma_idesc_bf16(128, K, 0, 1);
    uint32_t fph = 0;
    bool ok = true;
    for (int it = 0; it < p.max_rounds && ok; ++it) {
      int s = 0;
      auto next = [&](int q) { return q + 1 == C::NSLOT ? 0 : q + 1; };
      for (int c = 0; c < C::KCH && ok; ++c) {
        const int s0 = s, s1 = next(s0), s2 = next(s1);
        s = next(s2);
        ok = mbar_wait(bar_full + 8 * s0, (fph >> s0) & 1u, abort_flag, p.status) &&
             mbar_wait(bar_full + 8 * s1, (fph >> s1) & 1u, abort_flag, p.status);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fph ^= (1u << s0) | (1u << s1);
        tc_fence_after();
        const uint32_t alo = umma_desc_lo(sm_u + s0 * C::SLOT);
        if (elect_one()) {
          const uint32_t blo = umma_desc_lo(sm_u + s1 * C::SLOT, 8192);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int mh = 0; mh < C::HALVES; ++mh)
              tc_mma_lo(tmem_base + mh * K, alo + mh * 1024 + kk * 2, blo + kk * 128, idesc, (c | kk) != 0 ? 1u : 0u);
          tc_commit(bar_empty + 8 * s1);
        }
        __syncwarp();
        ok = __all_sync(0xffffffffu, mbar_wait(bar_full + 8 * s2, (fph >> s2) & 1u, abort_flag, p.status));
        if (!ok) break;
        fph ^= 1u << s2;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t blo = umma_desc_lo(sm_u + s2 * C::SLOT, 8192);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int mh = 0; mh < C::HALVES; ++mh) tc_mma_lo(tmem_base + mh * K, alo + mh * 1024 + kk * 2, blo + kk * 128, idesc, 1u);
          tc_commit(bar_empty + 8 * s0);
          tc_commit(bar_empty + 8 * s2);
          if (c == C::KCH - 1) tc_commit(bar_acc);
        }
        __syncwarp();
      }
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar_r, it & 1u, abort_flag, p.status));
      if (!ok) break;
      tc_fence_after();
      for (int c = 0; c < C::KCH && ok; ++c) {
        const int sl = c % C::NRING;
        ok = __all_sync(0xffffffffu, mbar_wait(bar_full + 8 * sl, (fph >> sl) & 1u, abort_flag, p.status));
        if (!ok) break;
        fph ^= 1u << sl;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t alo = umma_desc_lo(sm_u + sl * C::SLOT), blo = umma_desc_lo(sR + c * C::SLOT, 8192);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int mh = 0; mh < C::HALVES; ++mh)
              tc_mma_lo(tmem_base + mh * K, alo + mh * 1024 + kk * 2, blo + kk * 128, idesc, (c | kk) != 0 ? 1u : 0u);
          tc_commit(bar_empty + 8 * sl);
          if (c == C::KCH - 1) tc_commit(bar_acc);
        }
        __syncwarp();
      }
      if (!ok || it == p.max_rounds - 1 || residual2() <= p.gate2) break;
      // the next round's first product overwrites the accumulators that the epilogue of this one reads
      ok = __all_sync(0xffffffffu, mbar_wait(bar_x, it & 1u, abort_flag, p.status));
      tc_fence_after();
    }
  } else {
    // ---------------------------------------------------------------- epilogues: 32 x 32 tiles
    const int q = warp & 3, ew = warp - 2, part = ew >> 2;
    constexpr int CPH = K / 32, NU = C::HALVES * CPH / 4;  // column tiles per accumulator, tiles per warp
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
    uint8_t* wbuf = smem + ew * C::EPI_WARP_BYTES;
    const uint32_t tB = smem_u32(wbuf), tF = tB + 8192;
    const uint32_t bc0 = bar_c0 + 16 * ew;
    uint32_t accph = 0, c0ph = 0;
    bool ok = true;
    auto tile_of = [&](int i, int& mh, int& ch) { const int c2 = part + i * 4; mh = c2 / CPH; ch = c2 - mh * CPH; };
    for (int it = 0; it < p.max_rounds && ok; ++it) {
      ok = __all_sync(0xffffffffu, mbar_wait(bar_acc, accph, abort_flag, p.status));
      accph ^= 1u;
      if (!ok) break;
      tc_fence_after();
      float sq4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int i = 0; i < NU; ++i) {
        int mh, ch;
        tile_of(i, mh, ch);
        const int l = mh * 128 + q * 32 + lane, col0 = ch * 32;
        float v[32];
        tc_ld32(taddr + mh * K + col0, v);
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          v[e] = ((col0 + e == l) ? 1.f : 0.f) - v[e];
          sq4[e & 3] = fmaf(v[e], v[e], sq4[e & 3]);
        }
        // row l, columns col0 .. col0 + 31: four 16-byte pieces of one 128-byte swizzled row
        const uint32_t rowp = sR + (l >> 6) * C::SLOT + (col0 >> 6) * 8192 + (l & 63) * 128;
        const int c16 = (col0 & 63) >> 3;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          uint32_t h[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            h[j] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[8 * w + 2 * j])) |
                   ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[8 * w + 2 * j + 1])) << 16);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(rowp + (((c16 + w) ^ (l & 7)) << 4)), "r"(h[0]), "r"(h[1]),
                       "r"(h[2]), "r"(h[3])
                       : "memory");
        }
      }
      double sq = (double)((sq4[0] + sq4[1]) + (sq4[2] + sq4[3]));
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (lane == 0) red[ew] = sq;
      fence_proxy_async_smem_tb();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_r);
      ok = __all_sync(0xffffffffu, mbar_wait(bar_r, it & 1u, abort_flag, p.status));
      if (!ok) break;
      const double r2 = residual2();
      const bool last = (r2 <= p.gate2) || it == p.max_rounds - 1;
      if (last && threadIdx.x == 64 && !(r2 <= p.accept2)) *not_converged = 1;
      ok = __all_sync(0xffffffffu, mbar_wait(bar_acc, accph, abort_flag, p.status));
      accph ^= 1u;
      if (!ok) break;
      tc_fence_after();
      // X += X R: old hi + lo tiles arrive one tile ahead, the new ones leave from the same buffer
      if (lane == 0) {
        int mh, ch;
        tile_of(0, mh, ch);
        mbar_expect_tx(bc0, 4096);
        tma_load_3d(tB, &maps.xhl, ch * 32, row_b + mh * 128 + q * 32, 0, bc0);
      }
#pragma unroll 1
      for (int i = 0; i < NU && ok; ++i) {
        int mh, ch;
        tile_of(i, mh, ch);
        const int row0 = row_b + mh * 128 + q * 32, col0 = ch * 32;
        const uint32_t buf = i & 1, tH = tB + buf * 4096, tL = tH + 2048;
        float v[32];
        tc_ld32(taddr + mh * K + col0, v);
        ok = __all_sync(0xffffffffu, mbar_wait(bc0 + 8 * buf, (c0ph >> buf) & 1u, abort_flag, p.status));
        if (!ok) break;
        c0ph ^= 1u << buf;
        const int sw2 = (lane >> 1) & 3;  // 64-byte rows, 16-byte pieces XOR-swizzled by (row / 2) mod 4
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t off = lane * 64 + ((c ^ sw2) << 4);
          uint32_t h[4], l[4];
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3]) : "r"(tH + off));
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(l[0]), "=r"(l[1]), "=r"(l[2]), "=r"(l[3]) : "r"(tL + off));
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            v[8 * c + 2 * j] += __uint_as_float(h[j] << 16) + __uint_as_float(l[j] << 16);
            v[8 * c + 2 * j + 1] += __uint_as_float(h[j] & 0xFFFF0000u) + __uint_as_float(l[j] & 0xFFFF0000u);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float x0 = v[8 * c + 2 * j], x1 = v[8 * c + 2 * j + 1];
            const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
            h[j] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
            l[j] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x0 - __bfloat162float(h0))) |
                   ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x1 - __bfloat162float(h1))) << 16);
          }
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tH + off), "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3]) : "memory");
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tL + off), "r"(l[0]), "r"(l[1]), "r"(l[2]), "r"(l[3]) : "memory");
        }
        // the stores of the previous tile have read their shared memory: its buffer takes the next old tile, and the
        // fp32 tile can be overwritten
        if (lane == 0) {
          tma_store_wait_read();
          if (i + 1 < NU) {
            int mh2, ch2;
            tile_of(i + 1, mh2, ch2);
            const uint32_t bn = bc0 + 8 * (buf ^ 1u);
            mbar_expect_tx(bn, 4096);
            tma_load_3d(tB + (buf ^ 1u) * 4096, &maps.xhl, ch2 * 32, row_b + mh2 * 128 + q * 32, 0, bn);
          }
        }
        __syncwarp();
        if (last) {
          if (want_c) {
            // column sums of squares over the tile's 32 rows: a transposing reduction leaves column `lane` in each lane
            float t2[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) t2[e] = v[e] * v[e];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
              for (int e = 0; e < o; ++e) {
                const float keep = (lane & o) ? t2[e + o] : t2[e], send = (lane & o) ? t2[e] : t2[e + o];
                t2[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
              }
            }
            atomicAdd(&cn[col0 + lane], t2[0]);
          }
          const int sw = lane & 7;
#pragma unroll
          for (int c = 0; c < 8; ++c)
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(tF + lane * 128 + ((c ^ sw) << 4)), "f"(v[4 * c]),
                         "f"(v[4 * c + 1]), "f"(v[4 * c + 2]), "f"(v[4 * c + 3])
                         : "memory");
        }
        fence_proxy_async_smem_tb();
        __syncwarp();
        if (lane == 0) {
          tma_store_3d(&maps.xhl, tH, col0, row0, 0);
          if (last) tma_store_2d(&maps.x, tF, col0, row0);
          tma_store_commit();
        }
      }
      if (lane == 0) tma_store_wait_all();
      tc_fence_before();
      __syncwarp();
      if (!ok || last) break;
      if (lane == 0) {
        asm volatile("fence.proxy.async;" ::: "memory");
        mbar_arrive(bar_x);
      }
      __syncwarp();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_free(tmem_base, C::TMEM_COLS);
  }
  if (*abort_flag) return;
  const size_t off = (size_t)b * K * K;
  if (*not_converged) {
    // a change of the transform that the rounds could not follow (or a singular block): elimination
    if (threadIdx.x == 0 && p.redo_count) atomicAdd(p.redo_count, 1);
    float* X = p.X + off;
    asm volatile("fence.proxy.async;" ::: "memory");  // (the bulk stores to X are complete; this thread's view of it follows)
    for (int e = threadIdx.x; e < K * K; e += C::THREADS) X[e] = __uint_as_float((uint32_t)p.A[off + e] << 16);
    if (!gauss_jordan(X, K, reinterpret_cast<float*>(smem), p.status)) return;
    for (int t = threadIdx.x; t < K; t += C::THREADS) {
      float c = 0.f;
      for (int i = 0; i < K; ++i) {
        const float x = X[(size_t)i * K + t];
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        p.hi[off + (size_t)i * K + t] = __bfloat16_as_ushort(h);
        p.lo[off + (size_t)i * K + t] = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(h)));
        c = fmaf(x, x, c);
      }
      cn[t] = c;
    }
    __syncthreads();
  }
  pdl_release();
  if (want_c) {
    float* cw = p.cw[prob];
    for (int t = threadIdx.x; t < K; t += C::THREADS) {
      float v = cn[t];
      p.c[(size_t)b * K + t] = v;
      if (cw) {
        const int g = p.g[prob], col = (b - p.blk0[prob]) * K + t;
        if (g % 32 == 0) {  // (whole warps: K is a multiple of 32)
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) atomicAdd(&cw[col / g], v);
        } else {
          atomicAdd(&cw[col / g], v);
        }
      }
    }
  }
}

template <int K>
static int ns_block_launch_t(cudaStream_t st, const NsMaps& maps, int nb, const NsParams& p, bool overlap) {
  using C = NsCfg<K>;
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(ns_block_kernel<K>, C::SMEM, done)) return CAFEQ_ERR_CUDA;
  launch_pdl_if(overlap, ns_block_kernel<K>, nb, C::THREADS, C::SMEM, st, maps, p);
  return CAFEQ_OK;
}

// hi and lo splits [nb * k, k] as the two planes of one 3-D view (lo must lie a multiple of 16 bytes after hi)
static bool make_map_hl(CUtensorMap* m, const uint16_t* hi, const uint16_t* lo, long long rows, int k) {
  EncodeTiledFn enc = get_encode_tiled();
  if (!enc || lo <= hi || (((uintptr_t)lo - (uintptr_t)hi) & 15)) return false;
  cuuint64_t dims[3] = {(cuuint64_t)k, (cuuint64_t)rows, 2};
  cuuint64_t strides[2] = {(cuuint64_t)k * 2, (cuuint64_t)((uintptr_t)lo - (uintptr_t)hi)};
  cuuint32_t box[3] = {32, 32, 2};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(hi), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A, hi, lo: bf16 [nb * k, k]; X: fp32 [nb, k, k] (written, not read)
static int ns_block_launch(cudaStream_t st, const uint16_t* A, uint16_t* hi, uint16_t* lo, float* X, int nb, int k, NsParams p, bool overlap) {
  NsMaps m;
  p.A = A; p.hi = hi; p.lo = lo; p.X = X;
  const long long rows = (long long)nb * k;
  if (!make_map_bf16(&m.a, A, k, rows, k, k) || !make_map_bf16(&m.xh_mn, hi, k, rows, k, 64) || !make_map_bf16(&m.xl_mn, lo, k, rows, k, 64) ||
      !make_map_bf16(&m.xh_k, hi, k, rows, k, k) || !make_map_hl(&m.xhl, hi, lo, rows, k) ||
      !make_map_2d(&m.x, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, X, k, rows, k, 32, 32, CU_TENSOR_MAP_SWIZZLE_128B))
    return CAFEQ_ERR_UNSUPPORTED;
  return k == 256 ? ns_block_launch_t<256>(st, m, nb, p, overlap) : ns_block_launch_t<128>(st, m, nb, p, overlap);
}

// hi = A^T, lo = 0: the cold start X0 = A^T of the iteration (A is bf16, so hi carries it exactly); 32 x 32 tiles
__global__ void __launch_bounds__(256) ns_cold_start_kernel(const uint16_t* A, int k, uint16_t* __restrict__ hi,
                                                            uint16_t* __restrict__ lo, const int32_t* status) {
  pdl_enter();
  if (cta_stopped(status)) return;
  __shared__ uint16_t tile[32][34];
  const size_t base = (size_t)blockIdx.z * k * k;
  const int j0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
  uint16_t v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) v[r] = A[base + (size_t)(i0 + threadIdx.y + 8 * r) * k + j0 + threadIdx.x];
#pragma unroll
  for (int r = 0; r < 4; ++r) tile[threadIdx.y + 8 * r][threadIdx.x] = v[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const size_t o = base + (size_t)(j0 + threadIdx.y + 8 * r) * k + i0 + threadIdx.x;
    hi[o] = tile[threadIdx.x][threadIdx.y + 8 * r];
    lo[o] = 0;
  }
}

// ------------------------------------------------------------------------------------------------
// Two chained three-term products of one block with the intermediate kept in shared memory as hi / lo splits:
//   KK_MINV_PATH:  grad -= (X^T G) X^T     X = M^-1 (hi / lo splits in memory), G = dL/dM^-1: either dense fp32, or for
//                  Eq. 4 formed here, G[l][j] = scale X[l][j] A_j; the sixteen epilogue warps split it into the operand
//                  layout while the tensor core works on the previous 64 rows of it
//   KK_PENALTY:    R = M M^T - I with ||R||_F^2,  out = R M
// What bounds it: one block's operands (1 MB at k = 256) enter one SM at 60 - 75 GB/s from L2, beside 13 us of products.
// As separate launches (form G, split it, two products) the splits and the intermediate made the trip through memory
// and every launch paid its own fill and drain.  Measured (106 blocks of 256): M^-1 path 36 us against 8.5 + 15 + 2 x 20;
// 72 blocks of 128: 10.7 us against 4.4 + 2 x 9.5.
// The intermediate T of k = 256 does not fit in shared memory as a whole (256 KB): its accumulators fill tensor memory,
// each 128-row half is split into shared memory in turn and the second product of that half reuses its columns.
// Shared memory: T area (4 slots; the split rows of G use it before T exists, two stages of hi + lo) + ring.
// ------------------------------------------------------------------------------------------------
enum { KK_MINV_PATH = 0, KK_PENALTY = 1 };

struct ChainMaps {
  CUtensorMap a1[2];  // hi / lo, first product: KK_MINV_PATH boxes of 64 x 64, KK_PENALTY boxes of K rows x 64
  CUtensorMap b2[2];  // hi / lo, second product: KK_MINV_PATH boxes of K rows x 64, KK_PENALTY boxes of 64 x 64
  CUtensorMap out;    // fp32, boxes of 32 x 32 (KK_MINV_PATH: read and written)
};
struct ChainParams {
  // KK_MINV_PATH: blocks below blk0[n] belong to problems that scale X (blk0[p] <= b < blk0[p + 1]); the others are dense
  int n;
  int blk0[KK_MAX_PROBS + 1];
  const float* A[KK_MAX_PROBS];     // per transformed index, or
  const float* Agrp[KK_MAX_PROBS];  // per group of g transformed indices
  int g[KK_MAX_PROBS];
  float scale[KK_MAX_PROBS];
  const float* X;                   // fp32 X
  const float* G;                   // fp32 dense G
  // KK_PENALTY
  double* sq;                       // ||R_b||_F^2 is added to sq[b * sq_stride]
  int sq_stride;
  int want_out;                     // 0: only the norms
  int32_t* status;
};

template <int K>
struct ChainCfg {
  static constexpr int HALVES = K / 128;
  static constexpr int KCH = K / 64;
  static constexpr int SLOT = K * 128;
  static constexpr int NRING = (K == 256) ? 3 : 8;
  static constexpr int NSLOT = NRING + 4;
  static constexpr int EPI_WARPS = 16;
  static constexpr int NBAR = 2 * NRING + 4 + 2 + 2 * EPI_WARPS;
  static constexpr int SMEM = 1024 + NSLOT * SLOT + 8 * NBAR + 64;
  static constexpr int TMEM_COLS = HALVES * K;
  static constexpr int THREADS = 64 + 32 * EPI_WARPS;
};

// fp32 -> hi / lo of 8 consecutive values
__device__ __forceinline__ void split8(const float* x, uint32_t* h, uint32_t* l) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat16 h0 = __float2bfloat16_rn(x[2 * j]), h1 = __float2bfloat16_rn(x[2 * j + 1]);
    h[j] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
    l[j] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x[2 * j] - __bfloat162float(h0))) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x[2 * j + 1] - __bfloat162float(h1))) << 16);
  }
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint32_t* v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}

template <int K, int MODE>
__global__ void __launch_bounds__(ChainCfg<K>::THREADS, 1)
kk_chain_kernel(const __grid_constant__ ChainMaps maps, const __grid_constant__ ChainParams p) {
  pdl_enter();
  using C = ChainCfg<K>;
  const bool raised = status_raised(p.status);  // (awaited at the end of the set-up)
  const int b = blockIdx.x, row_b = b * K;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + C::NSLOT * C::SLOT);
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8 * C::NRING;
  const uint32_t bar_gfull = bar_empty + 8 * C::NRING;  // two stages of G
  const uint32_t bar_gempty = bar_gfull + 16;
  const uint32_t bar_acc = bar_gempty + 16;             // a product is complete
  const uint32_t bar_t = bar_acc + 8;                   // a half of T is in shared memory
  const uint32_t bar_c0 = bar_t + 8;                    // two per epilogue warp
  uint32_t* tmem_slot = (uint32_t*)(bars + C::NBAR);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sm_u = smem_u32(smem);
  const uint32_t sT = sm_u, sRing = sm_u + 4 * C::SLOT;
  const bool second = MODE == KK_MINV_PATH || p.want_out;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&maps.a1[0]);
    tma_prefetch_desc(&maps.a1[1]);
    tma_prefetch_desc(&maps.b2[0]);
    tma_prefetch_desc(&maps.b2[1]);
    for (int s = 0; s < C::NRING; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar_gfull + 8 * s, C::EPI_WARPS);
      mbar_init(bar_gempty + 8 * s, 1);
    }
    mbar_init(bar_acc, 1);
    mbar_init(bar_t, C::EPI_WARPS);
    for (int s = 0; s < 2 * C::EPI_WARPS; ++s) mbar_init(bar_c0 + 8 * s, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)C::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  const bool stopped = __syncthreads_or(raised) != 0;
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (stopped) {
    if (warp == 1) tmem_free(tmem_base, C::TMEM_COLS);
    return;
  }

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer: hi and lo of every 64-entry chunk
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      const int rounds = second ? 1 + C::HALVES : 1;
      for (int r = 0; r < rounds && ok; ++r) {
        const bool kmajor = (MODE == KK_MINV_PATH) == (r > 0);  // boxes of K rows x 64 entries, or of 64 x 64
        for (int c = 0; c < C::KCH && ok; ++c)
          for (int u = 0; u < 2; ++u, ++it) {
            const uint32_t s = it % C::NRING, ph = (it / C::NRING) & 1u;
            if (!mbar_wait(bar_empty + 8 * s, ph ^ 1u, abort_flag, p.status)) { ok = false; break; }
            mbar_expect_tx(bar_full + 8 * s, C::SLOT);
            const CUtensorMap* m = r ? &maps.b2[u] : &maps.a1[u];
            const uint32_t dst = sRing + s * C::SLOT;
            if (kmajor) {
              tma_load_2d(dst, m, c * 64, row_b, bar_full + 8 * s);
            } else {
              for (int j = 0; j < K / 64; ++j) tma_load_2d(dst + j * 8192, m, j * 64, row_b + c * 64, bar_full + 8 * s);
            }
          }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (converged warp, one elected lane)
    uint32_t it = 0;
    bool ok = true;
    auto wait_full = [&](uint32_t i) {
      return __all_sync(0xffffffffu, mbar_wait(bar_full + 8 * (i % C::NRING), (i / C::NRING) & 1u, abort_flag, p.status)) != 0;
    };
    // first product: k x k, three terms
    for (int c = 0; c < C::KCH && ok; ++c, it += 2) {
      const uint32_t sh = it % C::NRING, sl = (it + 1) % C::NRING;
      if constexpr (MODE == KK_MINV_PATH) {
        ok = __all_sync(0xffffffffu, mbar_wait(bar_gfull + 8 * (c & 1), (c >> 1) & 1u, abort_flag, p.status)) && wait_full(it);
        if (!ok) break;
        tc_fence_after();
        constexpr uint32_t idesc = umma_idesc_bf16(128, K, 1, 1);
        const uint32_t gh = umma_desc_lo(sT + (c & 1) * 2 * C::SLOT, 8192), gl = gh + (C::SLOT >> 4);
        if (elect_one()) {
          const uint32_t xh = umma_desc_lo(sRing + sh * C::SLOT, 8192);
#pragma unroll
          for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
              for (int mh = 0; mh < C::HALVES; ++mh)
                tc_mma_lo(tmem_base + mh * K, xh + mh * 1024 + kk * 128, (t ? gl : gh) + kk * 128, idesc, (c | t | kk) != 0 ? 1u : 0u);
          tc_commit(bar_empty + 8 * sh);
        }
        __syncwarp();
        ok = wait_full(it + 1);
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t xl = umma_desc_lo(sRing + sl * C::SLOT, 8192);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int mh = 0; mh < C::HALVES; ++mh)
              tc_mma_lo(tmem_base + mh * K, xl + mh * 1024 + kk * 128, gh + kk * 128, idesc, 1u);
          tc_commit(bar_empty + 8 * sl);
          tc_commit(bar_gempty + 8 * (c & 1));
          if (c == C::KCH - 1) tc_commit(bar_acc);
        }
        __syncwarp();
      } else {
        ok = wait_full(it) && wait_full(it + 1);
        if (!ok) break;
        tc_fence_after();
        constexpr uint32_t idesc = umma_idesc_bf16(128, K, 0, 0);
        if (elect_one()) {
          const uint32_t mhi = umma_desc_lo(sRing + sh * C::SLOT), mlo = umma_desc_lo(sRing + sl * C::SLOT);
#pragma unroll
          for (int t = 0; t < 3; ++t)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
              for (int mh = 0; mh < C::HALVES; ++mh)
                tc_mma_lo(tmem_base + mh * K, (t == 1 ? mlo : mhi) + mh * 1024 + kk * 2, (t == 2 ? mlo : mhi) + kk * 2, idesc,
                          (c | t | kk) != 0 ? 1u : 0u);
          tc_commit(bar_empty + 8 * sh);
          tc_commit(bar_empty + 8 * sl);
          if (c == C::KCH - 1) tc_commit(bar_acc);
        }
        __syncwarp();
      }
    }
    // second product: one 128-row half of T at a time
    constexpr int BMN = (MODE == KK_MINV_PATH) ? 0 : 1;
    constexpr uint32_t idesc2 = umma_idesc_bf16(128, K, 0, BMN);
    constexpr uint32_t bstep = BMN ? 128 : 2, lbo = BMN ? 8192 : 16;
    for (int h = 0; h < C::HALVES && ok && second; ++h) {
      ok = __all_sync(0xffffffffu, mbar_wait(bar_t, h & 1u, abort_flag, p.status));
      tc_fence_after();
      for (int c = 0; c < C::KCH && ok; ++c, it += 2) {
        const uint32_t sh = it % C::NRING, sl = (it + 1) % C::NRING;
        const uint32_t th = umma_desc_lo(sT + c * 16384), tl = th + (C::KCH * 16384 >> 4);
        ok = wait_full(it);
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t bh = umma_desc_lo(sRing + sh * C::SLOT, lbo);
#pragma unroll
          for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              tc_mma_lo(tmem_base + h * K, (t ? tl : th) + kk * 2, bh + kk * bstep, idesc2, (c | t | kk) != 0 ? 1u : 0u);
          tc_commit(bar_empty + 8 * sh);
        }
        __syncwarp();
        ok = wait_full(it + 1);
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t bl = umma_desc_lo(sRing + sl * C::SLOT, lbo);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) tc_mma_lo(tmem_base + h * K, th + kk * 2, bl + kk * bstep, idesc2, 1u);
          tc_commit(bar_empty + 8 * sl);
          if (c == C::KCH - 1) tc_commit(bar_acc);
        }
        __syncwarp();
      }
    }
  } else {
    // ---------------------------------------------------------------- splitting of G, splitting of T, output
    const int q = warp & 3, ew = warp - 2, part = ew >> 2;
    const int et = threadIdx.x - 64;
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
    bool ok = true;
    if constexpr (MODE == KK_MINV_PATH) {
      // a thread owns 8 consecutive columns (the same ones in every row it touches)
      constexpr int CG = K / 8, NI = 64 * CG / (32 * C::EPI_WARPS);
      const int cg = et % CG, r0 = et / CG;
      constexpr int RSTEP = 32 * C::EPI_WARPS / CG;
      int prob = -1;
      for (int q2 = 0; q2 < p.n; ++q2)
        if (b >= p.blk0[q2] && b < p.blk0[q2 + 1]) prob = q2;
      float mul[8];
      const float* src = (prob >= 0 ? p.X : p.G) + (size_t)b * K * K + cg * 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) mul[j] = 1.f;
      if (prob >= 0) {
        const int t0 = (b - p.blk0[prob]) * K + cg * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          mul[j] = p.scale[prob] * (p.Agrp[prob] ? p.Agrp[prob][(t0 + j) / p.g[prob]] : p.A[prob][t0 + j]);
      }
      float4 nx[NI][2];
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const float4* s4 = reinterpret_cast<const float4*>(src + (size_t)(r0 + i * RSTEP) * K);
        nx[i][0] = s4[0];
        nx[i][1] = s4[1];
      }
#pragma unroll 1
      for (int c = 0; c < C::KCH && ok; ++c) {
        const uint32_t gb = sT + (c & 1) * 2 * C::SLOT;
        ok = __all_sync(0xffffffffu, mbar_wait(bar_gempty + 8 * (c & 1), ((c >> 1) & 1u) ^ 1u, abort_flag, p.status));
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int r = r0 + i * RSTEP;
          const float x[8] = {nx[i][0].x * mul[0], nx[i][0].y * mul[1], nx[i][0].z * mul[2], nx[i][0].w * mul[3],
                              nx[i][1].x * mul[4], nx[i][1].y * mul[5], nx[i][1].z * mul[6], nx[i][1].w * mul[7]};
          uint32_t h[4], l[4];
          split8(x, h, l);
          const uint32_t o = gb + (cg >> 3) * 8192 + r * 128 + (((cg & 7) ^ (r & 7)) << 4);
          sts128(o, h);
          sts128(o + C::SLOT, l);
        }
        if (c + 1 < C::KCH) {
#pragma unroll
          for (int i = 0; i < NI; ++i) {
            const float4* s4 = reinterpret_cast<const float4*>(src + (size_t)((c + 1) * 64 + r0 + i * RSTEP) * K);
            nx[i][0] = s4[0];
            nx[i][1] = s4[1];
          }
        }
        fence_proxy_async_smem_tb();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_gfull + 8 * (c & 1));
      }
    }
    constexpr int CPH = K / 32;
    double sq = 0.0;
    for (int h = 0; h < C::HALVES && ok; ++h) {
      // h = 0: T is complete; later: the second product of the previous half has finished reading the T area
      if (h == 0 || second) ok = __all_sync(0xffffffffu, mbar_wait(bar_acc, h & 1u, abort_flag, p.status));
      if (!ok) break;
      tc_fence_after();
      float sq4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int ch = part; ch < CPH; ch += 4) {
        const int m = q * 32 + lane, col0 = ch * 32;
        float v[32];
        tc_ld32(taddr + h * K + col0, v);
        if constexpr (MODE == KK_PENALTY) {
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            if (col0 + e == h * 128 + m) v[e] -= 1.f;
            sq4[e & 3] = fmaf(v[e], v[e], sq4[e & 3]);
          }
        }
        if (second) {
          const uint32_t rowp = sT + (col0 >> 6) * 16384 + m * 128;
          const int c16 = (col0 & 63) >> 3;
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            uint32_t hh[4], ll[4];
            split8(v + 8 * w, hh, ll);
            const uint32_t o = rowp + (((c16 + w) ^ (m & 7)) << 4);
            sts128(o, hh);
            sts128(o + C::KCH * 16384, ll);
          }
        }
      }
      if constexpr (MODE == KK_PENALTY) sq += (double)((sq4[0] + sq4[1]) + (sq4[2] + sq4[3]));
      fence_proxy_async_smem_tb();
      tc_fence_before();
      __syncwarp();
      if (lane == 0 && second) mbar_arrive(bar_t);
    }
    if constexpr (MODE == KK_PENALTY) {
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (ok && lane == 0 && sq != 0.0) atomicAdd(p.sq + (long long)b * p.sq_stride, sq);
    }
    if (ok && second) ok = __all_sync(0xffffffffu, mbar_wait(bar_acc, C::HALVES & 1u, abort_flag, p.status));
    if (ok && second) {
      tc_fence_after();
      const uint32_t tB = sm_u + ew * 8192, bc0 = bar_c0 + 16 * ew;  // two fp32 tiles per warp (every slot is free now)
      constexpr int NU = C::HALVES * CPH / 4;
      auto tile_of = [&](int i, int& mh, int& ch) { const int c2 = part + i * 4; mh = c2 / CPH; ch = c2 - mh * CPH; };
      const int sw = lane & 7;
      if (MODE == KK_MINV_PATH && lane == 0) {
        int mh, ch;
        tile_of(0, mh, ch);
        mbar_expect_tx(bc0, 4096);
        tma_load_2d(tB, &maps.out, ch * 32, row_b + mh * 128 + q * 32, bc0);
      }
#pragma unroll 1
      for (int i = 0; i < NU && ok; ++i) {
        int mh, ch;
        tile_of(i, mh, ch);
        const uint32_t t = tB + (i & 1) * 4096;
        float v[32];
        tc_ld32(taddr + mh * K + ch * 32, v);
        if constexpr (MODE == KK_MINV_PATH) {
          ok = __all_sync(0xffffffffu, mbar_wait(bc0 + 8 * (i & 1), (i >> 1) & 1u, abort_flag, p.status));
          if (!ok) break;
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            float4 x;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w)
                         : "r"(t + lane * 128 + ((c ^ sw) << 4)));
            v[4 * c] = x.x - v[4 * c];
            v[4 * c + 1] = x.y - v[4 * c + 1];
            v[4 * c + 2] = x.z - v[4 * c + 2];
            v[4 * c + 3] = x.w - v[4 * c + 3];
          }
        }
        if (lane == 0) {
          tma_store_wait_read();  // the previous tile's store has read the other buffer
          if (MODE == KK_MINV_PATH && i + 1 < NU) {
            int mh2, ch2;
            tile_of(i + 1, mh2, ch2);
            const uint32_t bn = bc0 + 8 * ((i + 1) & 1);
            mbar_expect_tx(bn, 4096);
            tma_load_2d(tB + ((i + 1) & 1) * 4096, &maps.out, ch2 * 32, row_b + mh2 * 128 + q * 32, bn);
          }
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c)
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(t + lane * 128 + ((c ^ sw) << 4)), "f"(v[4 * c]),
                       "f"(v[4 * c + 1]), "f"(v[4 * c + 2]), "f"(v[4 * c + 3])
                       : "memory");
        fence_proxy_async_smem_tb();
        __syncwarp();
        if (lane == 0) {
          tma_store_2d(&maps.out, t, ch * 32, row_b + mh * 128 + q * 32);
          tma_store_commit();
        }
      }
      if (lane == 0) tma_store_wait_all();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_free(tmem_base, C::TMEM_COLS);
  }
}

template <int K, int MODE>
static int kk_chain_launch_t(cudaStream_t st, const ChainMaps& maps, int nb, const ChainParams& p, bool overlap) {
  using C = ChainCfg<K>;
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(kk_chain_kernel<K, MODE>, C::SMEM, done)) return CAFEQ_ERR_CUDA;
  launch_pdl_if(overlap, kk_chain_kernel<K, MODE>, nb, C::THREADS, C::SMEM, st, maps, p);
  return CAFEQ_OK;
}

// hi, lo: splits of X (KK_MINV_PATH) or M (KK_PENALTY), bf16 [nb * k, k]; out fp32 [nb, k, k]
static int kk_chain_launch(cudaStream_t st, int mode, const uint16_t* hi, const uint16_t* lo, float* out, int nb, int k,
                           const ChainParams& p, bool overlap = true) {
  ChainMaps m;
  const long long rows = (long long)nb * k;
  const int box1 = mode == KK_MINV_PATH ? 64 : k, box2 = mode == KK_MINV_PATH ? k : 64;
  if (!make_map_bf16(&m.a1[0], hi, k, rows, k, box1) || !make_map_bf16(&m.a1[1], lo, k, rows, k, box1) ||
      !make_map_bf16(&m.b2[0], hi, k, rows, k, box2) || !make_map_bf16(&m.b2[1], lo, k, rows, k, box2) ||
      !make_map_2d(&m.out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, out, k, rows, k, 32, 32, CU_TENSOR_MAP_SWIZZLE_128B))
    return CAFEQ_ERR_UNSUPPORTED;
  if (mode == KK_MINV_PATH) return k == 256 ? kk_chain_launch_t<256, KK_MINV_PATH>(st, m, nb, p, overlap) : kk_chain_launch_t<128, KK_MINV_PATH>(st, m, nb, p, overlap);
  return k == 256 ? kk_chain_launch_t<256, KK_PENALTY>(st, m, nb, p, overlap) : kk_chain_launch_t<128, KK_PENALTY>(st, m, nb, p, overlap);
}

}  // namespace cafeq
