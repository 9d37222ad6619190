// Dense products on CTA pairs (cta_group::2, M = 256): C = alpha * sum_t A_t B_t^T + beta * C0 + gamma * I over bf16 splits, for
// matrices that fill the chip with tiles of 256 x (up to 256).
//
//   * Every distinct array of a split is loaded once per 64-wide contraction chunk, whatever the number of terms that use it
//     (three terms: four arrays instead of six; six terms: six instead of twelve): 43 bytes per cycle and SM instead of the 96 of
//     a 128 x 256 tile on one SM with its own loads per term.
//   * The leading term hi * hi and the small terms have an accumulator each (2 x 256 of 512 tensor-memory columns), summed in
//     the epilogue.  Every addition to an accumulator is rounded at the accumulator's size, so small terms added to the large
//     sum would cost as much accuracy as the large ones.
//   * Two products with the same right operand and shape can share a launch (the two symmetric iterates of the Gram iteration);
//     a symmetric result is computed on and above the diagonal tiles and stored on both sides.
#pragma once

#include "kernels_gemm.cuh"
#include "kernels_pair_mma.cuh"
#include "pair_rules.cuh"

namespace cafeq {

constexpr int T2_SLOT = 16384;  // one array's 128 rows x 64 contraction entries
constexpr int T2_NSLOT = 12;    // stages of na + nb slots each
constexpr int T2_MAX_ARR = 3, T2_MAX_TERMS = 6;
constexpr int T2_SMEM = 1024 + T2_NSLOT * T2_SLOT + 512;

// the terms of a product over split arrays, and its tiles
struct T2Shape {
  int bn;         // tile columns, a multiple of 32 (of 128 with an MN-major B)
  int tm, tn;     // tiles
  int sym;        // the results are symmetric: tiles on and above the diagonal, Chi / Clo also mirrored (M = N, bn = 256)
  int na, nb, nterms;
  int nstage;     // T2_NSLOT / (na + nb)
  int two;        // terms with ac = 1 have the second accumulator
  int split;      // the product is one part of a contraction: alpha times it is stored in C, nothing else is done
  int8_t ta[T2_MAX_TERMS], tb[T2_MAX_TERMS], ac[T2_MAX_TERMS];
};
struct T2Maps {
  CUtensorMap a[2][T2_MAX_ARR];  // per product of the launch
  CUtensorMap b[T2_MAX_ARR];
};
struct T2Params {
  TgParams p[2];  // the products of the launch: same M, N, K, operands per a[0], a[1]
  int nprob;
  T2Shape sh;
};

struct T2Cta {
  uint8_t* smem;
  uint32_t bar_full, bar_empty, bar_acc;  // full: signalled and awaited in the leader
  uint32_t tmem;
  uint32_t rank;
  volatile int* abort_flag;
};

// Set-up of a CTA pair; false: the launch is to be left at once (nothing held).
__device__ __forceinline__ bool t2_enter(T2Cta& c, uint8_t* smem_raw, bool raised) {
  c.smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(c.smem + T2_NSLOT * T2_SLOT);
  c.bar_full = smem_u32(bars);
  c.bar_empty = c.bar_full + 8 * T2_NSLOT;
  c.bar_acc = c.bar_empty + 8 * T2_NSLOT;
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * T2_NSLOT + 1);
  c.abort_flag = (volatile int*)(tmem_slot + 1);
  c.rank = cluster_rank();
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < T2_NSLOT / 2; ++s) {
      mbar_init(c.bar_full + 8 * s, 1);
      mbar_init(c.bar_empty + 8 * s, 1);
    }
    mbar_init(c.bar_acc, 1);
    *c.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(tmem_slot), 512u);
  tc_fence_before();
  const bool stopped = pair_stopped(raised, tmem_slot + 2);
  tc_fence_after();
  c.tmem = *tmem_slot;
  if (stopped && warp == 1) tmem_free_pair(c.tmem, 512u);
  return !stopped;
}

// The scale path of the straight-through gradient as a product's epilogue: with v = d loss / d Uhat (the product times alpha) and the
// residual Delta = hi + lo, coef = sign(usel) / a * sum over the group of v Delta.  The product itself is not stored.  Records are
// group-major.
struct T2Ste {
  const uint16_t *hi, *lo;  // [M, ld]
  long long ld;
  const float *a, *usel;    // [groups, M]
  float* coef;
  int g;                    // 64 or 128
};

// Where a tile of a batched or split product lies: corner of its operands, first chunk and number of chunks of its contraction,
// batch (of the output).
struct T2At {
  int ax, ay, bx, by, c0, nc, b;
};

// One tile of one product, by all threads of both CTAs.  sq_acc: where the sum of squares goes (p.sq only says that there is
// one).  chunks / tiles: contraction chunks and tiles this pair has done before
// in this launch (the barriers' phases).  On return both CTAs are done with each other's shared memory.
__device__ __forceinline__ void t2_tile(const T2Cta& cta, const CUtensorMap* ma, const CUtensorMap* mb, const TgParams& p,
                                        const T2Shape& sh, double* sq_acc, const int ti, const int tj, const T2At at,
                                        const uint32_t chunks, const uint32_t tiles, const T2Ste* ste = nullptr, const bool meets = false) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta.rank, base = smem_u32(cta.smem);
  const int bn = sh.bn, bh = bn >> 1, narr = sh.na + sh.nb;
  const int m0 = ti * 256 + (int)rank * 128, n0 = tj * bn;  // this CTA's accumulator rows; the tile's columns
  const int kchunks = at.nc, nstage = sh.nstage;
  uint32_t s = chunks % nstage, ph = (chunks / nstage) & 1u;

  if (warp == 0) {
    if (lane == 0) {
      const int a_mn = p.a_mn, b_mn = p.b_mn;
      const int nrow = n0 + (int)rank * bh;  // this CTA's half of the B rows
      for (int c = 0; c < kchunks; ++c) {
        const int l0 = (at.c0 + c) * TG_BK;
        if (!mbar_wait(cta.bar_empty + 8 * s, ph ^ 1u, cta.abort_flag, p.status)) break;
        if (rank == 0) mbar_expect_tx(cta.bar_full + 8 * s, 2 * (sh.na * T2_SLOT + sh.nb * bh * 128));
        const uint32_t bar = cluster_addr(cta.bar_full + 8 * s, 0);
        uint32_t dst = base + s * narr * T2_SLOT;
        for (int u = 0; u < sh.na; ++u, dst += T2_SLOT) {
          if (a_mn) {
            for (int j = 0; j < 2; ++j) tma_load_pair(dst + j * 8192, ma + u, at.ax + m0 + j * 64, at.ay + l0, bar);
          } else {
            tma_load_pair(dst, ma + u, at.ax + l0, at.ay + m0, bar);
          }
        }
        for (int u = 0; u < sh.nb; ++u, dst += T2_SLOT) {
          if (b_mn) {
            for (int j = 0; j < bh / 64; ++j) tma_load_pair(dst + j * 8192, mb + u, at.bx + nrow + j * 64, at.by + l0, bar);
          } else {
            tma_load_pair(dst, mb + u, at.bx + l0, at.by + nrow, bar);
          }
        }
        if (++s == (uint32_t)nstage) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = umma_idesc_bf16(256, bn, p.a_mn, p.b_mn);
      const uint32_t astep = p.a_mn ? 128 : 2, bstep = p.b_mn ? 128 : 2;  // 16 contraction entries further, in 16-byte units
      const uint32_t albo = p.a_mn ? 8192 : 16, blbo = p.b_mn ? 8192 : 16;
      for (int c = 0; c < kchunks; ++c) {
        if (!__all_sync(0xffffffffu, mbar_wait(cta.bar_full + 8 * s, ph, cta.abort_flag, p.status))) break;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t sa = base + s * narr * T2_SLOT, sb = sa + sh.na * T2_SLOT;
          // The terms in their order and in reverse by turns: a product on another accumulator than the one before it costs some
          // 90 cycles, once per chunk instead of twice.
          uint32_t used = c ? 3u : 0u;  // accumulators written so far
          for (int i = 0; i < sh.nterms; ++i) {
            const int t = (c & 1) ? sh.nterms - 1 - i : i;
            const uint32_t ac = sh.ac[t], d = cta.tmem + ac * 256u;
            const uint32_t alo = umma_desc_lo(sa + sh.ta[t] * T2_SLOT, albo), blo = umma_desc_lo(sb + sh.tb[t] * T2_SLOT, blbo);
            const uint32_t acc = (used >> ac) & 1u;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) tc_mma_pair(d, alo + kk * astep, blo + kk * bstep, idesc, kk ? 1u : acc);
            used |= 1u << ac;
          }
          // (one barrier per chunk and direction: with one per array the issuing warp's waits, some 400 cycles each, set the pace)
          tc_commit_pair(cta.bar_empty + 8 * s);
          if (c == kchunks - 1) tc_commit_pair(cta.bar_acc);
        }
        __syncwarp();
        if (++s == (uint32_t)nstage) { s = 0; ph ^= 1u; }
      }
    }
  } else {
    const int q = warp & 3, part = (warp - 2) >> 2;
    bool ok = mbar_wait(cta.bar_acc, tiles & 1u, cta.abort_flag, p.status);
    ok = __all_sync(0xffffffffu, ok);
    float sum = 0.f, av = 0.f, us = 0.f;  // scale path: over this warp's 64 columns; the group's record
    const int row = m0 + q * 32 + lane;
    float* half = reinterpret_cast<float*>(cta.smem) + (part >> 1) * 128 + q * 32;
    if (ok) {
      tc_fence_after();
      const uint32_t taddr = cta.tmem + ((uint32_t)(q * 32) << 16);
      // a mirrored store of a diagonal tile would write what the tile itself writes
      uint16_t* th = sh.sym ? (ti != tj ? p.Chi : nullptr) : p.Cthi;
      uint16_t* tl = sh.sym ? (ti != tj ? p.Clo : nullptr) : p.Ctlo;
      double sq = 0.0;
      float* tile = reinterpret_cast<float*>(cta.smem + (warp - 2) * 4608);  // [32][36] per warp (the slots are free now)
      if (ste) {
        // this warp's 64 of 256 columns: a group of 64, or with the next warp one of 128
        const int col = at.b * 256 + part * 64;
        const bool rv = row < p.M;
        if (rv) {
          av = ste->a[(long long)(col / ste->g) * p.M + row];
          us = ste->usel[(long long)(col / ste->g) * p.M + row];
        }
#pragma unroll 1
        for (int c8 = 0; c8 < 4; ++c8) {  // 16 columns
          const long long o = (long long)row * ste->ld + col + c8 * 16;
          uint4 h[2], l[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            h[j] = l[j] = make_uint4(0u, 0u, 0u, 0u);
            if (rv) {
              h[j] = ld_plain(reinterpret_cast<const uint4*>(ste->hi + o) + j);
              l[j] = ld_plain(reinterpret_cast<const uint4*>(ste->lo + o) + j);
            }
          }
          float v[16], u[16];
          tc_ld16(taddr + part * 64 + c8 * 16, v);
          tc_ld16(taddr + 256u + part * 64 + c8 * 16, u);
          const uint32_t* hw = reinterpret_cast<const uint32_t*>(h);
          const uint32_t* lw = reinterpret_cast<const uint32_t*>(l);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            sum = fmaf(v[2 * e] + u[2 * e], __uint_as_float(hw[e] << 16) + __uint_as_float(lw[e] << 16), sum);
            sum = fmaf(v[2 * e + 1] + u[2 * e + 1], __uint_as_float(hw[e] & 0xFFFF0000u) + __uint_as_float(lw[e] & 0xFFFF0000u), sum);
          }
        }
        sum *= p.alpha;
        if (ste->g == 128 && (part & 1)) half[lane] = sum;
      } else if (sh.split) {
        // part of a contraction (M, N multiples of 32; C and its pitch of 16 bytes)
#pragma unroll 1
        for (int ch = part; ch < bn / 32; ch += TG_EPI_PARTS) {
          if (n0 + ch * 32 >= p.N || m0 + q * 32 >= p.M) break;
          float v[32];
          tc_ld32(taddr + ch * 32, v);
          if (sh.two) {
            float u[32];
            tc_ld32(taddr + 256u + ch * 32, u);
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] += u[e];
          }
#pragma unroll
          for (int j = 0; j < 8; ++j)
            *reinterpret_cast<float4*>(tile + lane * 36 + 4 * j) =
                make_float4(p.alpha * v[4 * j], p.alpha * v[4 * j + 1], p.alpha * v[4 * j + 2], p.alpha * v[4 * j + 3]);
          __syncwarp();
          float* out = p.C + (long long)at.b * p.sCb + (long long)(m0 + q * 32 + (lane >> 3)) * p.ldc + n0 + ch * 32 + (lane & 7) * 4;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *reinterpret_cast<float4*>(out + (long long)(4 * i) * p.ldc) =
                *reinterpret_cast<const float4*>(tile + (i * 4 + (lane >> 3)) * 36 + (lane & 7) * 4);
          __syncwarp();
        }
      } else
#pragma unroll 1
      for (int ch = part; ch < bn / 32; ch += TG_EPI_PARTS)
        tg_epilogue_chunk(p, at.b, m0, n0, ch, taddr, sh.two ? taddr + 256u : 0u, th, tl, tile, q, lane, sq);
      if (p.sq) {
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0 && sq != 0.0) atomicAdd(sq_acc, (sh.sym && ti != tj) ? 2.0 * sq : sq);
      }
    }
    if (ste) {
      // The warps of a group of 128 meet whether or not their waits succeeded: this barrier has no limit of its own.
      __syncwarp();
      if (ste->g == 128) asm volatile("bar.sync %0, 64;" ::"r"(1 + (part >> 1) * 4 + q) : "memory");
      if (ok && row < p.M && (ste->g == 64 || !(part & 1))) {
        if (ste->g == 128) sum += half[lane];
        const float sgn = (us > 0.f) ? 1.f : ((us < 0.f) ? -1.f : 0.f);
        ste->coef[(long long)((at.b * 256 + part * 64) / ste->g) * p.M + row] = (av > 0.f) ? sgn * sum / av : 0.f;
      }
    }
  }
  // neither CTA goes on (or leaves) while the other's products may read its shared memory or signal its barriers (meets: the grid meets
  // next, which includes that)
  __syncwarp();
  tc_fence_before();
  if (meets) return;
  __syncthreads();
  cluster_sync();
  tc_fence_after();
}

__global__ void __launch_bounds__(TG_THREADS, 1)
tc_pair_gemm_kernel(const __grid_constant__ T2Maps maps, const __grid_constant__ T2Params tp) {
  pdl_enter();
  const bool raised = status_raised(tp.p[0].status);  // (awaited at the end of the set-up)
  if (tg_stopped(tp.p[0])) return;  // (the same answer in both CTAs: the residuals are those of earlier launches)
  extern __shared__ uint8_t smem_raw[];
  const T2Shape& sh = tp.sh;
  int t = (int)(blockIdx.x >> 1), ti, tj, prob;
  if (sh.sym) {
    const int per = sh.tm * (sh.tm + 1) / 2;
    prob = t / per;
    t -= prob * per;
    ti = 0;
    while (t >= sh.tm - ti) { t -= sh.tm - ti; ++ti; }
    tj = ti + t;
  } else {
    const int per = sh.tm * sh.tn;
    prob = t / per;
    t -= prob * per;
    tj = t / sh.tm;
    ti = t - tj * sh.tm;
  }
  if (threadIdx.x < sh.na + sh.nb) tma_prefetch_desc((int)threadIdx.x < sh.na ? &maps.a[prob][threadIdx.x] : &maps.b[threadIdx.x - sh.na]);
  T2Cta cta;
  if (!t2_enter(cta, smem_raw, raised)) return;
  t2_tile(cta, maps.a[prob], maps.b, tp.p[prob], sh, tp.p[prob].sq, ti, tj, T2At{0, 0, 0, 0, 0, tp.p[prob].K / TG_BK, 0}, 0, 0);
  if ((threadIdx.x >> 5) == 1) tmem_free_pair(cta.tmem, 512u);
}

// ------------------------------------------------------------------------------------------------
// The rest of the pseudo-inverse iteration in one launch: R = I - A X and X += X R by turns, one persistent pair per two SMs, a
// grid-wide barrier after each product (cooperative launch).  Well-conditioned matrices have ended before it and it returns at
// once: as launches of their own the iterations that are skipped took 2.3 us each, 0.25 ms a matrix.
// ------------------------------------------------------------------------------------------------
struct T2LoopMaps {
  CUtensorMap a[2][2];      // per product
  CUtensorMap b[3][2];      // product 0; product 1 with the transposed iterate in the first / second buffer
};
struct T2LoopParams {
  TgParams p[2][2];         // product, buffer of the transposed iterate that product 1 reads
  T2Shape sh[2];
  int it0, it1;             // iterations
  uint32_t* arrived;        // zero before the launch
};

// All CTAs of the grid, bounded; false: some CTA did not come (status raised).
__device__ __forceinline__ bool grid_meet(uint32_t* arrived, uint32_t target, volatile int* abort_flag, int32_t* status) {
  asm volatile("fence.proxy.async;" ::: "memory");  // what was stored (or lies in shared memory that is filled next) meets bulk copies
  __threadfence();
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    atomicAdd(arrived, 1u);
    const uint64_t t0 = global_timer_ns();
    while (*(volatile uint32_t*)arrived < target) {
      if (*abort_flag || global_timer_ns() - t0 > BD_WAIT_NS) {
        *abort_flag = 1;
        raise_status(status, CAFEQ_ERR_TIMEOUT);
        ok = false;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
  }
  ok = __syncthreads_and(ok) != 0;
  asm volatile("fence.proxy.async;" ::: "memory");
  return ok;
}

__global__ void __launch_bounds__(TG_THREADS, 1)
pinv_loop_kernel(const __grid_constant__ T2LoopMaps maps, const __grid_constant__ T2LoopParams lp) {
  pdl_enter();
  const bool raised = status_raised(lp.p[0][0].status);
  if (tg_stopped(lp.p[0][0], lp.it0)) return;
  extern __shared__ uint8_t smem_raw[];
  T2Cta cta;
  if (!t2_enter(cta, smem_raw, raised)) return;
  const int npairs = (int)(gridDim.x >> 1), pair = (int)(blockIdx.x >> 1);
  uint32_t chunks = 0, tiles = 0, met = 0;
  for (int it = lp.it0; it < lp.it1; ++it) {
    if (it > lp.it0 && tg_stopped(lp.p[0][0], it)) break;
    const int cur = it & 1;
    bool ok = true, done = false;
    for (int pr = 0; pr < 2 && ok; ++pr) {
      if (pr && (done = tg_stopped(lp.p[1][cur], it))) break;
      const TgParams& p = lp.p[pr][cur];
      const T2Shape& sh = lp.sh[pr];
      for (int t = pair; t < sh.tm * sh.tn; t += npairs) {
        const int tj = t / sh.tm;
        t2_tile(cta, maps.a[pr], maps.b[pr ? 1 + cur : 0], p, sh, p.sq + it, t - tj * sh.tm, tj,
                T2At{0, 0, 0, 0, 0, p.K / TG_BK, 0}, chunks, tiles, nullptr, t + npairs >= sh.tm * sh.tn);
        if (t + npairs < sh.tm * sh.tn) {  // the epilogue's scratch lies in the ring that bulk copies write next
          asm volatile("fence.proxy.async;" ::: "memory");
          __syncthreads();
        }
        chunks += p.K / TG_BK;
        ++tiles;
      }
      ok = grid_meet(lp.arrived, ++met * gridDim.x, cta.abort_flag, p.status);
      tc_fence_after();
    }
    if (!ok || done) break;
  }
  cluster_sync();
  if ((threadIdx.x >> 5) == 1) tmem_free_pair(cta.tmem, 512u);
}

// Batched 256 x 256 products with a long contraction (Gram matrices and operator gradients of blocks of 256): every pair takes a
// slice of one block's contraction (and one of `reps` column blocks that are summed) and stores its product as a part of its own;
// sum_parts_kernel adds a block's parts in their order, so that a call repeats itself bit for bit.  As tiles of 64 columns with
// the whole contraction each, 14 blocks had 112 CTAs with 64 chunks of three terms in a row, 66 us.  Straight-through gradient of the
// 9B-shaped v-o pair 792 -> 729 us (its parts added atomically, in no fixed order: 721).
__global__ void __launch_bounds__(TG_THREADS, 1)
tc_pair_split_kernel(const __grid_constant__ T2Maps maps, const __grid_constant__ TgParams p, const __grid_constant__ T2Shape sh,
                     const int reps, const int slices) {
  pdl_enter();
  const bool raised = status_raised(p.status);  // (awaited at the end of the set-up)
  extern __shared__ uint8_t smem_raw[];
  const int unit = (int)(blockIdx.x >> 1), s = unit % slices, rep = (unit / slices) % reps, b = unit / (slices * reps);
  const int all = (p.K + TG_BK - 1) / TG_BK, c0 = (int)((long long)s * all / slices), c1 = (int)((long long)(s + 1) * all / slices);
  if (threadIdx.x < sh.na + sh.nb) tma_prefetch_desc((int)threadIdx.x < sh.na ? &maps.a[0][threadIdx.x] : &maps.b[threadIdx.x - sh.na]);
  T2Cta cta;
  if (!t2_enter(cta, smem_raw, raised)) return;
  const int blk = b * reps + rep;
  t2_tile(cta, maps.a[0], maps.b, p, sh, nullptr, 0, 0,
          T2At{blk * p.colsA_per_batch, blk * p.rowsA_per_batch, blk * p.colsB_per_batch, blk * p.rowsB_per_batch, c0, c1 - c0, unit}, 0, 0);
  if ((threadIdx.x >> 5) == 1) tmem_free_pair(cta.tmem, 512u);
}

// out[b] = sum of its n parts, in their order (blocks of 256 x 256), and optionally its bf16 splits.  Four entries a thread (grid: 64 per
// block), the parts' loads in flight together; bound by reading the parts from L2.
__global__ void __launch_bounds__(256) sum_parts_kernel(const float* parts, int n, float* __restrict__ out, uint16_t* __restrict__ hi,
                                                        uint16_t* __restrict__ lo, const int32_t* status) {
  pdl_enter();
  if (cta_stopped(status)) return;
  const long long b = blockIdx.x >> 6;
  const int e = ((blockIdx.x & 63) * 256 + threadIdx.x) * 4;
  const float* p = parts + b * n * 65536 + e;
  float4 s = ld_plain(reinterpret_cast<const float4*>(p));
#pragma unroll 8
  for (int i = 1; i < n; ++i) {
    const float4 x = ld_plain(reinterpret_cast<const float4*>(p + (long long)i * 65536));
    s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
  }
  const long long o = b * 65536 + e;
  if (((uintptr_t)out & 15) == 0) {
    *reinterpret_cast<float4*>(out + o) = s;
  } else {  // (a caller's gradient at any float address)
    out[o] = s.x; out[o + 1] = s.y; out[o + 2] = s.z; out[o + 3] = s.w;
  }
  if (hi) {
    const float x[4] = {s.x, s.y, s.z, s.w};
    uint32_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __nv_bfloat16 t = __float2bfloat16_rn(x[j]);
      h[j] = __bfloat16_as_ushort(t);
      l[j] = __bfloat16_as_ushort(__float2bfloat16_rn(x[j] - __bfloat162float(t)));
    }
    *reinterpret_cast<uint2*>(hi + o) = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
    *reinterpret_cast<uint2*>(lo + o) = make_uint2(l[0] | (l[1] << 16), l[2] | (l[3] << 16));
  }
}

// Scale path of the straight-through gradient on blocks of 256: v = alpha * (hi + lo) N_b over the columns of block b, reduced to one
// coefficient per group in the epilogue.  4096 x 3584: the product stored as fp32, read again and reduced took 47 + 28 us.
__global__ void __launch_bounds__(TG_THREADS, 1)
tc_pair_ste_kernel(const __grid_constant__ T2Maps maps, const __grid_constant__ TgParams p, const __grid_constant__ T2Shape sh,
                   const __grid_constant__ T2Ste ste) {
  pdl_enter();
  const bool raised = status_raised(p.status);  // (awaited at the end of the set-up)
  extern __shared__ uint8_t smem_raw[];
  const int unit = (int)(blockIdx.x >> 1), b = unit / sh.tm, ti = unit - b * sh.tm;
  if (threadIdx.x < sh.na + sh.nb) tma_prefetch_desc((int)threadIdx.x < sh.na ? &maps.a[0][threadIdx.x] : &maps.b[threadIdx.x - sh.na]);
  T2Cta cta;
  if (!t2_enter(cta, smem_raw, raised)) return;
  t2_tile(cta, maps.a[0], maps.b, p, sh, nullptr, ti, 0, T2At{b * 256, 0, 0, b * 256, 0, 4, b}, 0, 0, &ste);
  if ((threadIdx.x >> 5) == 1) tmem_free_pair(cta.tmem, 512u);
}

static int t2_launch(cudaStream_t st, const T2Maps& maps, const T2Params& tp) {
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(tc_pair_gemm_kernel, T2_SMEM, done)) return CAFEQ_ERR_CUDA;
  const T2Shape& sh = tp.sh;
  launch_pairs_if(true, tc_pair_gemm_kernel, tp.nprob * (sh.sym ? sh.tm * (sh.tm + 1) / 2 : sh.tm * sh.tn), TG_THREADS, T2_SMEM, st,
                  maps, tp);
  return CAFEQ_OK;
}

// All pairs of the grid have to be resident: a cooperative launch, one pair for every two SMs at most.
static int pinv_loop_launch(cudaStream_t st, const T2LoopMaps& maps, const T2LoopParams& lp) {
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(pinv_loop_kernel, T2_SMEM, done)) return CAFEQ_ERR_CUDA;
  int pairs = 0;
  for (const T2Shape& sh : lp.sh) pairs = sh.tm * sh.tn > pairs ? sh.tm * sh.tn : pairs;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(TG_THREADS);
  cfg.dynamicSmemBytes = T2_SMEM;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int fit = 0;
  if (cudaOccupancyMaxActiveClusters(&fit, pinv_loop_kernel, &cfg) != cudaSuccess || fit < 1) return CAFEQ_ERR_CUDA;
  if (pairs > fit) cfg.gridDim = dim3(2 * fit);
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, pinv_loop_kernel, maps, lp) == cudaSuccess ? CAFEQ_OK : CAFEQ_ERR_CUDA;
}

// Products of M x N in tiles of 256 x bn over na and nb arrays: the terms A_i B_j with i + j < order, all but the leading one on the
// second accumulator.
static T2Shape t2_shape(int M, int N, int bn, int na, int nb, int order) {
  T2Shape s;
  memset(&s, 0, sizeof(s));
  s.bn = bn; s.tm = (M + 255) / 256; s.tn = (N + bn - 1) / bn;
  s.na = na; s.nb = nb;
  for (int d = 0; d < order; ++d)
    for (int i = 0; i <= d; ++i)
      if (i < na && d - i < nb) {
        s.ta[s.nterms] = (int8_t)i;
        s.tb[s.nterms] = (int8_t)(d - i);
        s.ac[s.nterms++] = d > 0;
      }
  s.two = s.nterms > 1;
  s.nstage = T2_NSLOT / (na + nb);
  return s;
}

// Slices of a contraction of length K in 74 / units parts, of 256 entries at least (a tile's fixed part is some 8 us).
static int t2_slices(int units, int K) {
  const int s = units < 74 ? 74 / units : 1, most = K / 256;
  return s < most ? s : (most > 0 ? most : 1);
}

// Dh / Dl: [M, nb * 256] (pitch ste.ld); Nh / Nl: blocks [nb * 256, 256]
static int tg_launch_ste(cudaStream_t st, const uint16_t* Nh, const uint16_t* Nl, int M, int nb, float alpha, const T2Ste& ste, int32_t* status) {
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(tc_pair_ste_kernel, T2_SMEM, done)) return CAFEQ_ERR_CUDA;
  T2Maps maps;
  memset(&maps, 0, sizeof(maps));
  const uint16_t* d[2] = {ste.hi, ste.lo};
  const uint16_t* n[2] = {Nh, Nl};
  for (int i = 0; i < 2; ++i)
    if (!make_map_bf16(&maps.a[0][i], d[i], nb * 256ll, M, ste.ld, 128) || !make_map_bf16(&maps.b[i], n[i], 256, nb * 256ll, 256, 128))
      return CAFEQ_ERR_UNSUPPORTED;
  TgParams p;
  memset(&p, 0, sizeof(p));
  p.M = M; p.N = 256; p.K = 256; p.batch = nb; p.divA = 1;
  p.alpha = alpha;
  p.status = status;
  const T2Shape sh = t2_shape(M, 256, 256, 2, 2, 2);
  launch_pairs_if(true, tc_pair_ste_kernel, nb * sh.tm, TG_THREADS, T2_SMEM, st, maps, p, sh, ste);
  return CAFEQ_OK;
}

// A: na arrays, B: nb arrays, each [rows, cols] with its pitch, either both stored with the contraction as rows (mn: [K, blocks * 256])
// or both with it as columns ([blocks * 256, K]).  Parts of alpha * sum over the column (row) blocks b * reps .. of A_b B_b^T: `count` of
// them for each of the `batch` blocks in a row, 65536 floats each (at most K / 256 * reps * batch of them; K >= 256).
static int tg_launch_split(cudaStream_t st, int na, const TgOperand* A, int nb, const TgOperand* B, int K, int batch, int reps, int mn,
                           float alpha, float* parts, int* count, int32_t* status) {
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(tc_pair_split_kernel, T2_SMEM, done)) return CAFEQ_ERR_CUDA;
  T2Maps maps;
  memset(&maps, 0, sizeof(maps));
  bool ok = true;
  for (int i = 0; i < na; ++i) ok = ok && make_map_bf16(&maps.a[0][i], A[i].ptr, A[i].cols, A[i].rows, A[i].pitch, mn ? 64 : 128);
  for (int i = 0; i < nb; ++i) ok = ok && make_map_bf16(&maps.b[i], B[i].ptr, B[i].cols, B[i].rows, B[i].pitch, mn ? 64 : 128);
  if (!ok) return CAFEQ_ERR_UNSUPPORTED;
  TgParams p;
  memset(&p, 0, sizeof(p));
  p.M = p.N = 256; p.K = K; p.batch = batch; p.divA = 1;
  p.a_mn = p.b_mn = mn;
  if (mn) p.colsA_per_batch = p.colsB_per_batch = 256;
  else p.rowsA_per_batch = p.rowsB_per_batch = 256;
  p.alpha = alpha;
  p.C = parts; p.ldc = 256; p.sCb = 65536;
  p.status = status;
  T2Shape sh = t2_shape(256, 256, 256, na, nb, na > nb ? na : nb);
  sh.split = 1;
  const int units = batch * reps, slices = t2_slices(units, K);
  *count = reps * slices;
  launch_pairs_if(true, tc_pair_split_kernel, units * slices, TG_THREADS, T2_SMEM, st, maps, p, sh, reps, slices);
  return CAFEQ_OK;
}

}  // namespace cafeq
