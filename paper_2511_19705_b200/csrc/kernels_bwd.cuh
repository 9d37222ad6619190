// Sparse backward of the transform pass on the tensor cores (tcgen05, sm_100a).
//
// Every (row, group) record of the forward pass carries a coefficient (dLoss / d group maximum, signed) and the
// position of the group's arg-max entry.  The gradient with respect to an operator block is a sum of outer
// products routed through those entries (Section 4.1: the group maximum is the only path from the transform
// to Eq. 4; App. D: the same for the LogSumExp surrogate):
//   input axis : gradT[B][i][j] = sum_o S[o][i] W[o, B k + j],   S[o][i] = coef(o, G) where i is the arg-max column of (o, G)
//   output axis: gradT[B][i][j] = sum_c S[i][c] W[B k + j, c],   S[i][c] = coef(B k + i, G(c)) where c is its arg-max column
// i.e. a dense k x k product whose left operand has one non-zero per (row, group).  The kernel streams the weight
// tiles once with TMA, writes the few non-zeros of S as a two-term bf16 split (hi + lo: fp32-grade coefficients)
// straight into shared memory in the swizzled operand layout, and accumulates the block gradient in tensor
// memory over all tiles of the block that the CTA owns; one flush per block and CTA adds it to global memory.
// The product is issued in the orientation (S^T W or W^T S) whose accumulator rows run along the fastest index of
// the requested output layout, so that the flush is coalesced atomic adds straight from registers.
//
// F16 form: when the caller holds an fp16 copy of the weights (W * 2^e, exact for every bf16 value that matters:
// fp16 keeps 11 significand bits against bf16's 8) the coefficients are written as ONE fp16 term (relative error
// 2^-12, scaled by a power of two so that the largest lands near 2^14) and the product is issued once instead of
// twice; the flush undoes both power-of-two scales.
//
// Several matrices can share one launch (see BwMulti): the tiles of all sub-problems form one list and every
// persistent CTA takes a contiguous run of it.
#pragma once

#include <cuda_fp16.h>

#include "kernels_fused.cuh"

namespace cafeq {

struct BwParams {
  int d_out, d_in;
  int g, ng;           // group width, groups per row
  int r;               // matrix blocks per operator block
  int n_major;         // blocks (input axis: column blocks; output axis: row blocks)
  int n_minor;         // tiles per block (input axis: of 64 rows, K = 256 of 128; output axis: of as many columns)
  int NG;              // groups of one row examined: input axis, those that meet 128 targets; output axis, those that meet a tile
  int gm;              // records are group-major (index = group * d_out + row) instead of row-major
  int transpose_out;   // store gradT[..][j][i]
  const float* coef;
  const int* idx;
  float* gradT;        // [n_major / r, k, k], accumulated with atomic adds (caller zeroes it)
  const float* coefmax;      // F16 form: device word holding max |coef| of this matrix (sets the coefficient scale)
  const float* w_inv_scale;  // F16 form: device word holding 2^-e of the fp16 weight copy
  const double* out_div;     // optional device word: the flushed gradient is divided by it (LogSumExp normaliser)
  int32_t* status;
};

constexpr int BW_MAX_SUB = 8;
struct BwMaps {
  CUtensorMap w[BW_MAX_SUB];
};
struct BwMulti {
  int n;
  int stream;  // as in BdMulti
  int tile_end[BW_MAX_SUB];
  BwParams p[BW_MAX_SUB];  // all share one status word
};

enum { BW_IN = 0, BW_OUT = 1 };
constexpr int BW_THREADS = 320;  // warp 0: TMA, warp 1: MMA, warps 2-9: operand builders and flush
constexpr int BW_NSTAGE = 3;
constexpr uint32_t BW_NONE = 0xFFFFFFFFu;

template <int F16>
struct BwCfg {  // K = 128
  static constexpr int K = 128;
  static constexpr int TERMS = F16 ? 1 : 2;
  static constexpr int NSTAGE = F16 ? 4 : BW_NSTAGE;
  static constexpr int STAGE_BYTES = K * 64 * 2;   // weight tile: 64 contraction entries x K
  static constexpr int S_TERM_BYTES = K * 64 * 2;  // S tile: K targets x 64 contraction entries, K-major, one 16-bit term
  static constexpr int S_BUF_BYTES = TERMS * S_TERM_BYTES;
  static constexpr int TMEM_COLS = K;
  static constexpr int RDEPTH = 4;  // records in flight per builder thread (8 bytes each, copied to shared memory ahead of their tile)
  static constexpr int REC_BYTES = RDEPTH * 256 * 8;
  static constexpr int SMEM = 1024 + NSTAGE * STAGE_BYTES + 2 * S_BUF_BYTES + REC_BYTES + 256;
};

// instruction descriptor for fp16 operands (format field 0), fp32 accumulation
__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N, int a_mn_major, int b_mn_major) {
  return (1u << 4) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// power of two that brings max |coef| just below 2^14 (fp16 holds up to 65504); 1 when there is nothing to scale
__device__ __forceinline__ float bw_coef_scale(const float* coefmax) {
  const float m = coefmax ? ld_plain(coefmax) : 0.f;
  if (!(m > 0.f) || !(m < 3.0e38f)) return 1.f;
  int e;
  frexpf(m, &e);  // m = f * 2^e, f in [0.5, 1)
  int sh = 14 - e;
  if (sh > 120) sh = 120;
  if (sh < -120) sh = -120;
  return exp2f((float)sh);
}

__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// byte offset of S[target][kk] inside one term of the S tile (128-byte rows, 16-byte chunks XOR-swizzled by the row index
// modulo 8; 64 contraction entries to a swizzle atom, the atoms of 128 targets 16 KB apart)
__device__ __forceinline__ uint32_t bw_s_offset(int target, int kk) {
  return (uint32_t)((kk >> 6) * 16384 + (target >> 3) * 1024 + (target & 7) * 128 + ((((kk >> 3) ^ target) & 7) << 4) + (kk & 7) * 2);
}

// SWAP = 0: accumulator rows = targets i, columns = j (coalesced when the output is stored transposed);
// SWAP = 1: rows = j, columns = i (coalesced for the plain layout).
template <int FORM, int SWAP, int F16>
__device__ __forceinline__ void bd_bwd_body(const BwMaps& maps, const BwMulti& mp, const int cta, const int ncta) {
  using C = BwCfg<F16>;
  constexpr int K = C::K;
  int32_t* const status = mp.p[0].status;
  const bool raised = status_raised(status);  // (awaited at the end of the set-up)
  const int total_tiles = mp.tile_end[mp.n - 1];
  const int t_begin = (int)(((long long)cta * total_tiles) / ncta);
  const int t_end = (int)(((long long)(cta + 1) * total_tiles) / ncta);
  if (t_begin >= t_end) return;
  int s_first = 0;
  while (mp.tile_end[s_first] <= t_begin) ++s_first;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sStage = smem;
  uint8_t* sS = smem + C::NSTAGE * C::STAGE_BYTES;
  uint8_t* sRec = sS + 2 * C::S_BUF_BYTES;
  uint64_t* bars = (uint64_t*)(sRec + C::REC_BYTES);
  // barrier slots: wfull[NSTAGE], wempty[NSTAGE], sfull[2], sempty[2], accf, acce
  const uint32_t bar_wfull = smem_u32(bars);
  const uint32_t bar_wempty = bar_wfull + 8 * C::NSTAGE;
  const uint32_t bar_sfull = bar_wempty + 8 * C::NSTAGE;
  const uint32_t bar_sempty = bar_sfull + 16;
  const uint32_t bar_accf = bar_sempty + 16;
  const uint32_t bar_acce = bar_accf + 8;
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * C::NSTAGE + 6);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&maps.w[s_first]);
    for (int s = 0; s < C::NSTAGE; ++s) {
      mbar_init(bar_wfull + 8 * s, 1);
      mbar_init(bar_wempty + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_sfull + 8 * b, 256);
      mbar_init(bar_sempty + 8 * b, 1);
    }
    mbar_init(bar_accf, 1);
    mbar_init(bar_acce, 256);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the S tiles start as zeros; afterwards the builders clear exactly what they wrote
  {
    uint4* z = reinterpret_cast<uint4*>(sS);
    for (int e = threadIdx.x; e < 2 * C::S_BUF_BYTES / 16; e += BW_THREADS) z[e] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
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
    // ---------------------------------------------------------------- TMA producer: one weight tile per stage
    if (lane == 0) {
      uint32_t it = 0;
      int sub = s_first;
      const uint64_t pol = l2_evict_first_policy();
      for (int gt = t_begin; gt < t_end; ++gt, ++it) {
        while (gt >= mp.tile_end[sub]) ++sub;
        const int tile = gt - (sub ? mp.tile_end[sub - 1] : 0);
        const int n_minor = mp.p[sub].n_minor;
        const CUtensorMap* tmW = &maps.w[sub];
        const int major = tile / n_minor, t = tile - major * n_minor;
        const uint32_t s = it % C::NSTAGE, ph = (it / C::NSTAGE) & 1u;
        if (!mbar_wait(bar_wempty + 8 * s, ph ^ 1u, abort_flag, status)) break;
        mbar_expect_tx(bar_wfull + 8 * s, C::STAGE_BYTES);
        const uint32_t dst = smem_u32(sStage + s * C::STAGE_BYTES);
        if constexpr (FORM == BW_IN) {
          // 64 rows x K columns as K / 64 boxes of 64 x 64 (one swizzle atom of the MN-major operand each)
          for (int n = 0; n < K / 64; ++n) {
            if (mp.stream) tma_load_2d_hint(dst + n * 8192, tmW, major * K + n * 64, t * 64, bar_wfull + 8 * s, pol);
            else tma_load_2d(dst + n * 8192, tmW, major * K + n * 64, t * 64, bar_wfull + 8 * s);
          }
        } else {
          // K rows x 64 columns: one box, K-major operand
          if (mp.stream) tma_load_2d_hint(dst, tmW, t * 64, major * K, bar_wfull + 8 * s, pol);
          else tma_load_2d(dst, tmW, t * 64, major * K, bar_wfull + 8 * s);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    // the whole warp runs the loop, one elected lane issues (see bd_pass_body)
    // the weight tile is MN-major on the input axis (contraction over its rows), K-major on the output axis
    constexpr int WMN = (FORM == BW_IN) ? 1 : 0;
    constexpr uint32_t idesc = F16 ? (SWAP ? umma_idesc_f16(128, K, WMN, 0) : umma_idesc_f16(128, K, 0, WMN))
                                   : (SWAP ? umma_idesc_bf16(128, K, WMN, 0) : umma_idesc_bf16(128, K, 0, WMN));
    constexpr uint32_t wlbo = (FORM == BW_IN) ? 8192 : 16, wstep = (FORM == BW_IN) ? 128 : 2;  // 16 contraction entries further
    const uint32_t sSt_u = smem_u32(sStage), sS_u = smem_u32(sS);
    auto wait_all = [&](uint32_t bar, uint32_t ph) { return __all_sync(0xffffffffu, mbar_wait(bar, ph, abort_flag, status)) != 0; };
    int sub = s_first, left = 0;  // tiles of the current block left in its list
    uint32_t run = 0, st = 0, sph = 0, it = 0;
    bool started = false;
    for (int gt = t_begin; gt < t_end; ++gt, ++it) {
      while (gt >= mp.tile_end[sub]) ++sub;
      const bool first = left == 0;
      if (first) {
        const int n_minor = mp.p[sub].n_minor, tile = gt - (sub ? mp.tile_end[sub - 1] : 0);
        left = n_minor - tile % n_minor;
        // the flush of the previous block must have drained the accumulators
        if (started) {
          if (!wait_all(bar_acce, (run - 1) & 1u)) break;
          tc_fence_after();
        }
        started = true;
      }
      const uint32_t b = it & 1u, bph = (it >> 1) & 1u;
      if (!wait_all(bar_wfull + 8 * st, sph)) break;
      if (!wait_all(bar_sfull + 8 * b, bph)) break;
      tc_fence_after();
      // last tile of this block in this CTA's run: hand the accumulators to the flush
      const bool last = --left == 0 || gt + 1 == t_end;
      if (elect_one()) {
        const uint32_t wlo = umma_desc_lo(sSt_u + st * C::STAGE_BYTES, wlbo);
#pragma unroll
        for (int term = 0; term < C::TERMS; ++term) {
          const uint32_t slo = umma_desc_lo(sS_u + b * C::S_BUF_BYTES + term * C::S_TERM_BYTES);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint32_t acc = (first && term == 0 && ks == 0) ? 0u : 1u;
            if constexpr (SWAP == 0) tc_mma_lo(tmem_base, slo + 2 * ks, wlo + ks * wstep, idesc, acc);
            else tc_mma_lo(tmem_base, wlo + ks * wstep, slo + 2 * ks, idesc, acc);
          }
        }
        tc_commit(bar_wempty + 8 * st);
        tc_commit(bar_sempty + 8 * b);
        if (last) tc_commit(bar_accf);
      }
      __syncwarp();
      if (last) ++run;
      if (++st == C::NSTAGE) { st = 0; sph ^= 1u; }
    }
  } else {
    // ---------------------------------------------------------------- operand builders (one record per thread and tile) and flush
    const int bt = threadIdx.x - 64;
    const int q = warp & 3, hw = (warp - 2) >> 2;
    // Position in the tile list, advanced without divisions: sub-problem, block, tile of the block.
    struct Cursor { int gt, sub, major, t; };
    auto advance = [&](Cursor& c) {
      ++c.gt;
      if (++c.t == mp.p[c.sub].n_minor) { c.t = 0; ++c.major; }
      if (c.gt == mp.tile_end[c.sub] && c.gt < total_tiles) { ++c.sub; c.major = c.t = 0; }
    };
    // This thread's record of a tile: address (-1: none), and where its entry of S goes.
    //   input axis: tile row bt & 63, group bt >> 6 of the block; column offset of that group inside the block
    //   output axis: block row bt; first column of the row's group minus the tile's first column
    auto rec_at = [&](const Cursor& c, int& colbase) -> long long {
      const BwParams& p = mp.p[c.sub];
      if constexpr (FORM == BW_IN) {
        const int rl = bt & 63, qq = bt >> 6;
        const int row = c.t * 64 + rl;
        const int G0 = (K >= p.g) ? c.major * p.NG : (c.major * K) / p.g;
        const int G = G0 + qq;
        colbase = G * p.g - c.major * K;
        if (qq >= p.NG || row >= p.d_out || G >= p.ng) return -1;
        return p.gm ? (long long)G * p.d_out + row : (long long)row * p.ng + G;
      } else {
        const int row = c.major * K + bt;
        const int G = (p.g == 64) ? c.t : ((p.g == 128) ? c.t >> 1 : (c.t * 64) / p.g);
        colbase = G * p.g - c.t * 64;
        if (bt >= K) return -1;
        return p.gm ? (long long)G * p.d_out + row : (long long)row * p.ng + G;
      }
    };
    // What bounds the builders: fence.proxy.async waits for every load that the thread has in flight, so a record that is
    // requested as a plain load ahead of the fence costs its whole memory latency once per tile (measured: 2100 cycles per
    // tile in the builders against 1400 for the tile's weights from HBM; 700 now, and the whole backward of a 9B-shaped
    // layer 133 -> 112 us, of a 27B-shaped one with groups of 64 371 -> 262 us).  Records are therefore copied to shared memory
    // with cp.async, RDEPTH tiles ahead; a thread reads only what it copied itself, so no barrier is involved. 
    uint8_t* const my_rec = sRec + bt * 8;
    Cursor ahead{};
    uint32_t pre = 0;          // tiles whose record has been requested
    auto request = [&]() {
      if (ahead.gt < t_end) {
        int cb;
        const long long pi = rec_at(ahead, cb);
        const BwParams& p = mp.p[ahead.sub];
        if (pi >= 0) {
          uint8_t* dst = my_rec + (pre % C::RDEPTH) * 2048;
          cp_async4(dst, p.coef + pi);
          cp_async4(dst + 4, p.idx + pi);
        }
        advance(ahead);
      }
      cp_async_commit();
      ++pre;
    };
    // record of the current tile, decoded: coefficient, target row, contraction index (tg < 0: none)
    auto take_rec = [&](const Cursor& c, uint32_t tl, float scale, float& cf, int& tg, int& kk) {
      tg = -1;
      int cb, ix;
      const long long pi = rec_at(c, cb);
      cp_async_wait<C::RDEPTH - 1>();
      asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=f"(cf), "=r"(ix) : "r"(smem_u32(my_rec) + (tl % C::RDEPTH) * 2048));
      if (pi < 0 || cf == 0.f) return;
      const int col = cb + ix;
      if constexpr (FORM == BW_IN) {
        if ((unsigned)col < (unsigned)K) { tg = col; kk = bt & 63; }
      } else {
        if ((unsigned)col < 64u) { tg = bt; kk = col; }
      }
      if constexpr (F16) cf *= scale;
    };
    // flush of one block: accumulators -> global memory, coalesced atomic adds straight from the registers
    // (accumulator row m = this thread's lane, 32 consecutive columns n per load)
    auto flush = [&](int sub, int major, uint32_t run) -> bool {
      const BwParams& p = mp.p[sub];
      bool okw = mbar_wait(bar_accf, run & 1u, abort_flag, status);
      okw = __all_sync(0xffffffffu, okw);
      if (!okw) return false;
      tc_fence_after();
      float mul = 1.f;
      if constexpr (F16) mul = (p.w_inv_scale ? ld_plain(p.w_inv_scale) : 1.f) / bw_coef_scale(p.coefmax);
      if (p.out_div) mul = (float)((double)mul / *p.out_div);
      float* out = p.gradT + (size_t)(major / p.r) * K * K;
      const int m = q * 32 + lane;
      for (int ch = 0; ch < 2; ++ch) {  // 32-column chunks per thread
        float v[32];
        const int n0 = hw * 64 + ch * 32;
        tc_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + n0, v);
#pragma unroll
        for (int c = 0; c < 32; ++c)
          if (v[c] != 0.f) atomicAdd(&out[(size_t)(n0 + c) * K + m], v[c] * mul);
      }
      tc_fence_before();
      mbar_arrive(bar_acce);
      return true;
    };

    uint32_t prevA = BW_NONE, prevB = BW_NONE;  // offsets this thread wrote into S buffer 0 / 1
    const int tile0 = t_begin - (s_first ? mp.tile_end[s_first - 1] : 0);
    Cursor cur{t_begin, s_first, tile0 / mp.p[s_first].n_minor, tile0 % mp.p[s_first].n_minor};
    ahead = cur;
    int cur_sub = s_first, cur_major = cur.major;
    uint32_t run = 0;
    bool ok = true;
    float scale = 1.f;
    if constexpr (F16) scale = bw_coef_scale(mp.p[s_first].coefmax);
    for (int i = 0; i < C::RDEPTH; ++i) request();
    for (uint32_t tl = 0; cur.gt < t_end && ok; ++tl) {
      const int sub = cur.sub, major = cur.major;
      if constexpr (F16) {
        if (sub != cur_sub) scale = bw_coef_scale(mp.p[sub].coefmax);
      }
      float cf;
      int tg, kk;
      take_rec(cur, tl, scale, cf, tg, kk);
      advance(cur);
      const uint32_t b = tl & 1u, sph = (tl >> 1) & 1u;
      if (major != cur_major || sub != cur_sub) {
        if (!flush(cur_sub, cur_major, run)) { ok = false; break; }
        ++run;
        cur_major = major;
        cur_sub = sub;
      }
      ok = mbar_wait(bar_sempty + 8 * b, sph ^ 1u, abort_flag, status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      uint8_t* buf = sS + b * C::S_BUF_BYTES;
      const uint32_t prev = b ? prevB : prevA;
      if (prev != BW_NONE) {
        *reinterpret_cast<uint16_t*>(buf + prev) = 0;
        if constexpr (!F16) *reinterpret_cast<uint16_t*>(buf + C::S_TERM_BYTES + prev) = 0;
      }
      uint32_t now = BW_NONE;
      if (tg >= 0) {
        now = bw_s_offset(tg, kk);
        if constexpr (F16) {
          *reinterpret_cast<uint16_t*>(buf + now) = __half_as_ushort(__float2half_rn(cf));
        } else {
          const __nv_bfloat16 hi = __float2bfloat16_rn(cf);
          const __nv_bfloat16 lo = __float2bfloat16_rn(cf - __bfloat162float(hi));
          *reinterpret_cast<uint16_t*>(buf + now) = __bfloat16_as_ushort(hi);
          *reinterpret_cast<uint16_t*>(buf + C::S_TERM_BYTES + now) = __bfloat16_as_ushort(lo);
        }
      }
      if (b) prevB = now; else prevA = now;
      fence_proxy_async_smem();
      mbar_arrive(bar_sfull + 8 * b);
      request();
    }
    if (ok) flush(cur_sub, cur_major, run);
  }

  // ---------------------------------------------------------------- teardown
  pdl_release();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_free(tmem_base, C::TMEM_COLS);
  }
}

// ------------------------------------------------------------------------------------------------
// K = 256 on CTA pairs (cta_group::2).  A tile is 128 contraction entries; each CTA holds half of the K columns (rows) of the weight
// tile and the S tile of 128 of the 256 targets, and 128 rows of the K x K accumulator.  That takes 256 of the 512 tensor-memory
// columns, so a block's sum is flushed by warps of its own while the next block is accumulated, and a pair flushes a block once where
// two CTAs did.  (One CTA with the whole accumulator in its tensor memory stood still during each flush: 15 of 91 us of a 9B-shaped
// layer.)  A tile holds eight products: every wait of the issuing warp costs it some 400 cycles.
// Both forms of a 9B-shaped layer, back to back: 102 us, issued by one elected lane of a converged warp 91, pairs 79, with the S tiles released
// at the scope of the cluster (relays, below) some 87.
// ------------------------------------------------------------------------------------------------
constexpr int BP_THREADS = 64 + 256 + 128 + 64;  // warp 0: TMA, warp 1: MMA, warps 2-9: operand builders, 10-13: flush, 14-15: relays

template <int F16>
struct BpCfg {
  static constexpr int TERMS = F16 ? 1 : 2;
  // A third S buffer, for one stage of the weights, where there is room: the relays (below) add more than a tile's time to an S tile's
  // way to the products.
  static constexpr int NSTAGE = F16 ? 3 : 2;
  static constexpr int NBUF = F16 ? 3 : 2;
  static constexpr int STAGE_BYTES = 32768;   // 128 contraction entries x 128 of K
  static constexpr int S_TERM_BYTES = 32768;  // 128 targets x 128 contraction entries, K-major, two swizzle atoms of 64 entries
  static constexpr int S_BUF_BYTES = TERMS * S_TERM_BYTES;
  static constexpr int RDEPTH = 4;
  static constexpr int REC_BYTES = RDEPTH * 256 * 8;
  static constexpr int SMEM = 1024 + NSTAGE * STAGE_BYTES + NBUF * S_BUF_BYTES + REC_BYTES + 256;
};

template <int FORM, int SWAP, int F16>
__device__ __forceinline__ void bd_bwd_pair_body(const BwMaps& maps, const BwMulti& mp, const int pair, const int npairs) {
  using C = BpCfg<F16>;
  constexpr int K = 256;
  int32_t* const status = mp.p[0].status;
  const bool raised = status_raised(status);  // (awaited at the end of the set-up)
  const int total_tiles = mp.tile_end[mp.n - 1];
  const int t_begin = (int)(((long long)pair * total_tiles) / npairs);
  const int t_end = (int)(((long long)(pair + 1) * total_tiles) / npairs);
  if (t_begin >= t_end) return;  // (the same in both CTAs)
  int s_first = 0;
  while (mp.tile_end[s_first] <= t_begin) ++s_first;
  const int rank = (int)cluster_rank();

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sStage = smem;
  uint8_t* sS = smem + C::NSTAGE * C::STAGE_BYTES;
  uint8_t* sRec = sS + C::NBUF * C::S_BUF_BYTES;
  uint64_t* bars = (uint64_t*)(sRec + C::REC_BYTES);
  // barrier slots: wfull[NSTAGE], wempty[NSTAGE], sfull[NBUF], sempty[NBUF], accf[2], acce[2]; wfull and acce are signalled by both CTAs
  // and awaited in the leader, sfull by the own builders (in the leader also by the other CTA's relay), the others are signalled in
  // both by the leader's commits
  const uint32_t bar_wfull = smem_u32(bars);
  const uint32_t bar_wempty = bar_wfull + 8 * C::NSTAGE;
  const uint32_t bar_sfull = bar_wempty + 8 * C::NSTAGE;
  const uint32_t bar_sempty = bar_sfull + 8 * C::NBUF;
  const uint32_t bar_accf = bar_sempty + 8 * C::NBUF;
  const uint32_t bar_acce = bar_accf + 16;
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * C::NSTAGE + 2 * C::NBUF + 4);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&maps.w[s_first]);
    for (int s = 0; s < C::NSTAGE; ++s) {
      mbar_init(bar_wfull + 8 * s, 1);
      mbar_init(bar_wempty + 8 * s, 1);
    }
    for (int b = 0; b < C::NBUF; ++b) {
      mbar_init(bar_sfull + 8 * b, rank == 0 ? 9 : 8);  // eight builder warps, the relay
      mbar_init(bar_sempty + 8 * b, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_accf + 8 * b, 1);
      mbar_init(bar_acce + 8 * b, 8);    // four flush warps of each CTA
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the S tiles start as zeros; afterwards the builders clear exactly what they wrote
  {
    uint4* z = reinterpret_cast<uint4*>(sS);
    for (int e = threadIdx.x; e < C::NBUF * C::S_BUF_BYTES / 16; e += BP_THREADS) z[e] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(tmem_slot), 512u);
  tc_fence_before();
  const bool stopped = pair_stopped(raised, tmem_slot + 2);
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (stopped) {
    if (warp == 1) tmem_free_pair(tmem_base, 512u);
    return;
  }

  // Relay of S buffer b (in the CTA that does not issue): the products that the leader issues read this CTA's S tiles, so the builders'
  // stores have to be released at the scope of the cluster.  That costs more than a tile's time (1 us), hence a warp for each buffer; from
  // a builder the arrival would wait for its records in flight too.  Step of a 9B-shaped layer: arrivals at the scope of the CTA, which do
  // not order those stores, 334 us; released by the builders 407, by one relay with two S buffers 352, with three 345, by a relay for each
  // of three 342.
  auto relay = [&](const uint32_t b) {
    if (b >= (uint32_t)C::NBUF || lane != 0) return;
    const uint32_t sfull0 = cluster_addr(bar_sfull, 0);
    uint32_t bph = 0;
    for (int gt = t_begin + (int)b; gt < t_end; gt += C::NBUF, bph ^= 1u) {
      if (!mbar_wait(bar_sfull + 8 * b, bph, abort_flag, status)) break;
      mbar_arrive_pair(sfull0 + 8 * b);
    }
  };
  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer: this CTA's half of one weight tile per stage
    if (lane == 0) {
      uint32_t s = 0, ph = 1;
      int sub = s_first;
      const uint64_t pol = l2_evict_first_policy();
      for (int gt = t_begin; gt < t_end; ++gt) {
        while (gt >= mp.tile_end[sub]) ++sub;
        const int tile = gt - (sub ? mp.tile_end[sub - 1] : 0);
        const int n_minor = mp.p[sub].n_minor;
        const CUtensorMap* tmW = &maps.w[sub];
        const int major = tile / n_minor, t = tile - major * n_minor;
        if (!mbar_wait(bar_wempty + 8 * s, ph, abort_flag, status)) break;
        if (rank == 0) mbar_expect_tx(bar_wfull + 8 * s, 2 * C::STAGE_BYTES);
        const uint32_t bar = cluster_addr(bar_wfull + 8 * s, 0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // boxes of 64 columns x 128 rows
          const uint32_t dst = smem_u32(sStage + s * C::STAGE_BYTES + h * 16384);
          const int x = (FORM == BW_IN) ? major * K + rank * 128 + h * 64 : t * 128 + h * 64;
          const int y = (FORM == BW_IN) ? t * 128 : major * K + rank * 128;
          if (mp.stream) tma_load_pair_hint(dst, tmW, x, y, bar, pol);
          else tma_load_pair(dst, tmW, x, y, bar);
        }
        if (++s == C::NSTAGE) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (the leader)
    if (rank == 0) {
      constexpr int WMN = (FORM == BW_IN) ? 1 : 0;
      constexpr uint32_t idesc = F16 ? (SWAP ? umma_idesc_f16(256, K, WMN, 0) : umma_idesc_f16(256, K, 0, WMN))
                                     : (SWAP ? umma_idesc_bf16(256, K, WMN, 0) : umma_idesc_bf16(256, K, 0, WMN));
      const uint32_t sSt_u = smem_u32(sStage), sS_u = smem_u32(sS);
      auto wait_all = [&](uint32_t bar, uint32_t ph) { return __all_sync(0xffffffffu, mbar_wait(bar, ph, abort_flag, status)) != 0; };
      int sub = s_first, left = 0;  // tiles of the current block left in its list
      uint32_t run = 0, st = 0, sph = 0, b = 0, bph = 0;
      for (int gt = t_begin; gt < t_end; ++gt) {
        while (gt >= mp.tile_end[sub]) ++sub;
        const bool first = left == 0;
        if (first) {
          const int n_minor = mp.p[sub].n_minor, tile = gt - (sub ? mp.tile_end[sub - 1] : 0);
          left = n_minor - tile % n_minor;
          // the flush of the block before the previous one must have drained this accumulator
          if (!wait_all(bar_acce + 8 * (run & 1u), ((run >> 1) & 1u) ^ 1u)) break;
          tc_fence_after();
        }
        if (!wait_all(bar_wfull + 8 * st, sph)) break;
        if (!__all_sync(0xffffffffu, mbar_wait_pair(bar_sfull + 8 * b, bph, abort_flag, status))) break;
        tc_fence_after();
        // last tile of this block in this pair's run: hand the accumulator to the flush
        const bool last = --left == 0 || gt + 1 == t_end;
        if (elect_one()) {
          const uint32_t d = tmem_base + (run & 1u) * 256u;
          const uint32_t wlo = umma_desc_lo(sSt_u + st * C::STAGE_BYTES, FORM == BW_IN ? 16384 : 16);
#pragma unroll
          for (int term = 0; term < C::TERMS; ++term) {
            const uint32_t slo = umma_desc_lo(sS_u + b * C::S_BUF_BYTES + term * C::S_TERM_BYTES);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              const uint32_t acc = (first && term == 0 && ks == 0) ? 0u : 1u;
              const uint32_t so = slo + (ks >> 2) * 1024 + (ks & 3) * 2;
              const uint32_t wo = wlo + (FORM == BW_IN ? ks * 128 : (ks >> 2) * 1024 + (ks & 3) * 2);
              tc_mma_pair(d, SWAP ? wo : so, SWAP ? so : wo, idesc, acc);
            }
          }
          tc_commit_pair(bar_wempty + 8 * st);
          tc_commit_pair(bar_sempty + 8 * b);
          if (last) tc_commit_pair(bar_accf + 8 * (run & 1u));
        }
        __syncwarp();
        if (last) ++run;
        if (++st == C::NSTAGE) { st = 0; sph ^= 1u; }
        if (++b == C::NBUF) { b = 0; bph ^= 1u; }
      }
    } else {
      relay(0);
    }
  } else if (warp < 10) {
    // ---------------------------------------------------------------- operand builders: one record per thread and tile
    const int bt = threadIdx.x - 64;
    const int rl = bt & 127, qq = bt >> 7;
    struct Cursor { int gt, sub, major, t; };
    auto advance = [&](Cursor& c) {
      ++c.gt;
      if (++c.t == mp.p[c.sub].n_minor) { c.t = 0; ++c.major; }
      if (c.gt == mp.tile_end[c.sub] && c.gt < total_tiles) { ++c.sub; c.major = c.t = 0; }
    };
    // This thread's record of a tile (-1: none) and the position of its group's first column.  128 columns count: on the input axis
    // this CTA's targets, on the output axis those of the tile; with NG = 2 thread qq has the group of their qq-th half (and what
    // falls there), else thread 0 the one group.  Input axis: tile row rl; output axis: target rl.
    auto rec_at = [&](const Cursor& c, int& colbase) -> long long {
      const BwParams& p = mp.p[c.sub];
      const int lo = (FORM == BW_IN) ? c.major * K + rank * 128 : c.t * 128;  // first of the 128 columns that count
      const int row = (FORM == BW_IN) ? c.t * 128 + rl : c.major * K + rank * 128 + rl;
      const int G = (p.g == 64) ? (lo >> 6) + qq : ((p.g == 128) ? lo >> 7 : (lo + qq * 64) / p.g);
      colbase = G * p.g - lo;
      if (qq >= p.NG || row >= p.d_out || G >= p.ng) return -1;
      return p.gm ? (long long)G * p.d_out + row : (long long)row * p.ng + G;
    };
    // Records are copied to shared memory RDEPTH tiles ahead (see bd_bwd_body); a thread reads only what it copied itself.
    uint8_t* const my_rec = sRec + bt * 8;
    const int tile0 = t_begin - (s_first ? mp.tile_end[s_first - 1] : 0);
    Cursor cur{t_begin, s_first, tile0 / mp.p[s_first].n_minor, tile0 % mp.p[s_first].n_minor};
    Cursor ahead = cur;
    uint32_t pre = 0;
    auto request = [&]() {
      if (ahead.gt < t_end) {
        int cb;
        const long long pi = rec_at(ahead, cb);
        const BwParams& p = mp.p[ahead.sub];
        if (pi >= 0) {
          uint8_t* dst = my_rec + (pre % C::RDEPTH) * 2048;
          cp_async4(dst, p.coef + pi);
          cp_async4(dst + 4, p.idx + pi);
        }
        advance(ahead);
      }
      cp_async_commit();
      ++pre;
    };
    uint32_t before[C::NBUF];  // offsets this thread wrote into each S buffer
#pragma unroll
    for (int i = 0; i < C::NBUF; ++i) before[i] = BW_NONE;
    uint32_t b = 0, bph = 1;
    int cur_sub = -1;
    float scale = 1.f;
    for (int i = 0; i < C::RDEPTH; ++i) request();
    for (uint32_t tl = 0; cur.gt < t_end; ++tl) {
      if constexpr (F16) {
        if (cur.sub != cur_sub) { scale = bw_coef_scale(mp.p[cur.sub].coefmax); cur_sub = cur.sub; }
      }
      const int sub = cur.sub;
      int cb, ix;
      float cf;
      const long long pi = rec_at(cur, cb);
      cp_async_wait<C::RDEPTH - 1>();
      asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=f"(cf), "=r"(ix) : "r"(smem_u32(my_rec) + (tl % C::RDEPTH) * 2048));
      advance(cur);
      const int col = cb + ix;
      const unsigned width = mp.p[sub].NG == 2 ? 64u : 128u;
      uint32_t now = BW_NONE;
      if (pi >= 0 && cf != 0.f && (unsigned)(col - qq * 64) < width) {
        const int tg = (FORM == BW_IN) ? col : rl, kk = (FORM == BW_IN) ? rl : col;
        now = bw_s_offset(tg, kk);
      }
      bool ok = mbar_wait(bar_sempty + 8 * b, bph, abort_flag, status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      uint8_t* buf = sS + b * C::S_BUF_BYTES;
      uint32_t prev = before[0];
#pragma unroll
      for (int i = 1; i < C::NBUF; ++i) prev = b == i ? before[i] : prev;
      if (prev != BW_NONE) {
        *reinterpret_cast<uint16_t*>(buf + prev) = 0;
        if constexpr (!F16) *reinterpret_cast<uint16_t*>(buf + C::S_TERM_BYTES + prev) = 0;
      }
      // (no other thread has this place to clear: it belongs to one row or target and one group, as the thread does)
      if (now != BW_NONE) {
        if constexpr (F16) {
          *reinterpret_cast<uint16_t*>(buf + now) = __half_as_ushort(__float2half_rn(cf * scale));
        } else {
          const __nv_bfloat16 hi = __float2bfloat16_rn(cf);
          const __nv_bfloat16 lo = __float2bfloat16_rn(cf - __bfloat162float(hi));
          *reinterpret_cast<uint16_t*>(buf + now) = __bfloat16_as_ushort(hi);
          *reinterpret_cast<uint16_t*>(buf + C::S_TERM_BYTES + now) = __bfloat16_as_ushort(lo);
        }
      }
#pragma unroll
      for (int i = 0; i < C::NBUF; ++i) before[i] = b == i ? now : before[i];
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_sfull + 8 * b);
      if (++b == C::NBUF) { b = 0; bph ^= 1u; }
      request();
    }
  } else if (warp >= 14) {
    if (rank != 0) relay(warp - 13);
  } else {
    // ---------------------------------------------------------------- flush: accumulators -> global memory, coalesced atomic adds
    const int q = warp & 3;
    const int m = rank * 128 + q * 32 + lane;
    const uint32_t acce0 = cluster_addr(bar_acce, 0);
    int sub = s_first;
    uint32_t run = 0;
    for (int gt = t_begin; gt < t_end; ++run) {
      while (gt >= mp.tile_end[sub]) ++sub;
      const BwParams& p = mp.p[sub];
      const int tile = gt - (sub ? mp.tile_end[sub - 1] : 0);
      const int major = tile / p.n_minor;
      gt += p.n_minor - (tile - major * p.n_minor);
      bool ok = mbar_wait(bar_accf + 8 * (run & 1u), (run >> 1) & 1u, abort_flag, status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      float mul = 1.f;
      if constexpr (F16) mul = (p.w_inv_scale ? ld_plain(p.w_inv_scale) : 1.f) / bw_coef_scale(p.coefmax);
      if (p.out_div) mul = (float)((double)mul / *p.out_div);
      float* out = p.gradT + (size_t)(major / p.r) * K * K + m;
#pragma unroll 1
      for (int ch = 0; ch < 8; ++ch) {
        float v[32];
        tc_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (run & 1u) * 256u + ch * 32, v);
        if (ch == 7) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_pair_tmem(acce0 + 8 * (run & 1u));
        }
#pragma unroll
        for (int c = 0; c < 32; ++c)
          if (v[c] != 0.f) atomicAdd(&out[(size_t)(ch * 32 + c) * K], v[c] * mul);
      }
    }
  }

  // ---------------------------------------------------------------- teardown
  pdl_release();
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // (neither CTA leaves while the other's products may read its shared memory)
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_free_pair(tmem_base, 512u);
  }
}

template <int K>
constexpr int bw_threads() { return K == 256 ? BP_THREADS : BW_THREADS; }
template <int K, int F16>
constexpr int bw_smem() {
  if constexpr (K == 256) return BpCfg<F16>::SMEM;
  else return BwCfg<F16>::SMEM;
}

template <int FORM, int K, int SWAP, int F16>
__global__ void __launch_bounds__(bw_threads<K>(), 1) bd_bwd_kernel(const __grid_constant__ BwMaps maps, const __grid_constant__ BwMulti mp) {
  pdl_wait();
  if constexpr (K == 256) bd_bwd_pair_body<FORM, SWAP, F16>(maps, mp, (int)blockIdx.x >> 1, (int)gridDim.x >> 1);
  else bd_bwd_body<FORM, SWAP, F16>(maps, mp, (int)blockIdx.x, (int)gridDim.x);
}

// Input-axis and output-axis matrices in one launch (fp16 single-term form): the first n_in CTAs run the input-axis
// list, the others the output-axis list.
template <int K, int SWAP_IN, int SWAP_OUT>
__global__ void __launch_bounds__(bw_threads<K>(), 1)
bd_bwd_dual_kernel(const __grid_constant__ BwMaps maps_in, const __grid_constant__ BwMulti mp_in,
                   const __grid_constant__ BwMaps maps_out, const __grid_constant__ BwMulti mp_out, const int n_in) {
  pdl_wait();
  if constexpr (K == 256) {
    const int pair = (int)blockIdx.x >> 1, n = (int)gridDim.x >> 1;
    if (pair < n_in) bd_bwd_pair_body<BW_IN, SWAP_IN, 1>(maps_in, mp_in, pair, n_in);
    else bd_bwd_pair_body<BW_OUT, SWAP_OUT, 1>(maps_out, mp_out, pair - n_in, n - n_in);
  } else {
    if ((int)blockIdx.x < n_in) bd_bwd_body<BW_IN, SWAP_IN, 1>(maps_in, mp_in, (int)blockIdx.x, n_in);
    else bd_bwd_body<BW_OUT, SWAP_OUT, 1>(maps_out, mp_out, (int)blockIdx.x - n_in, (int)gridDim.x - n_in);
  }
}

// host side ------------------------------------------------------------------------------------------------
static bool bw_supported(int axis_in, int d_out, int d_in, long long ld, int k, int g, const void* W) {
  if (!(k == 128 || k == 256)) return false;
  if ((ld % 8) || ((uintptr_t)W & 15)) return false;
  if (axis_in) {
    if (d_in % k) return false;
    if (!(k % g == 0 || g % k == 0)) return false;
    if (k / g > 4) return false;
  } else {
    if (d_out % k || d_in % 64 || g % 64 || d_in % g) return false;
  }
  return true;
}

static std::atomic<int> g_bw_min_tiles{6};  // tiles per CTA at least (more when problems overlap: see cafeq_set_overlap_mode)

// contraction entries of a tile
constexpr int bw_tile(int k) { return k == 256 ? 128 : 64; }
// rows of a weight box
constexpr int bw_box(int axis_in, int k) { return (k == 256 || !axis_in) ? 128 : 64; }

static void bw_fill_tiles(BwParams& p, int axis_in, int k) {
  const int rows = bw_tile(k);
  if (axis_in) {
    p.n_major = p.d_in / k;
    p.n_minor = (p.d_out + rows - 1) / rows;
    p.NG = (128 >= p.g) ? 128 / p.g : 1;  // (K = 256 has groups of 64 at least: two)
  } else {
    p.n_major = p.d_out / k;
    p.n_minor = (p.d_in + rows - 1) / rows;
    p.NG = (rows == 128 && p.g % 128) ? 2 : 1;
  }
}

template <int FORM, int K, int SWAP, int F16>
static int bw_launch_t(cudaStream_t st, const BwMaps& maps, BwMulti mp, int min_tiles) {
  constexpr int SMEM = bw_smem<K, F16>();
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(bd_bwd_kernel<FORM, K, SWAP, F16>, SMEM, done)) return CAFEQ_ERR_CUDA;
  // one persistent CTA per SM at most; small problems use fewer CTAs so that every CTA has several tiles per
  // flush (a flush moves k * k floats whatever the number of tiles behind it)
  long long total = 0, majors = 0;
  for (int s = 0; s < mp.n; ++s) {
    bw_fill_tiles(mp.p[s], FORM == BW_IN, K);
    total += (long long)mp.p[s].n_major * mp.p[s].n_minor;
    majors += mp.p[s].n_major;
    mp.tile_end[s] = (int)total;
  }
  for (int s = mp.n; s < BW_MAX_SUB; ++s) mp.tile_end[s] = (int)total;
  mp.stream = l2_stream(2.0 * bw_tile(K) * K * total);
  long long want = total / (min_tiles > 0 ? min_tiles : 1);
  if (want < majors) want = majors;
  if (want > total) want = total;
  constexpr int most = K == 256 ? 74 : 148;  // (pairs at K = 256)
  const int grid = want < most ? (int)want : most;
  if (K == 256) launch_pairs_if(true, bd_bwd_kernel<FORM, K, SWAP, F16>, grid, bw_threads<K>(), SMEM, st, maps, mp);
  else launch_pdl(bd_bwd_kernel<FORM, K, SWAP, F16>, grid, bw_threads<K>(), SMEM, st, maps, mp);
  return CAFEQ_OK;
}

static int bw_dispatch(cudaStream_t st, int axis_in, int k, int swap, int f16, const BwMaps& maps, const BwMulti& mp, int min_tiles) {
#define BW_CASE(AX, F, KK, SW, HF) \
  if ((axis_in != 0) == (AX) && k == KK && swap == SW && f16 == HF) return bw_launch_t<F, KK, SW, HF>(st, maps, mp, min_tiles);
  BW_CASE(true, BW_IN, 128, 0, 0)
  BW_CASE(true, BW_IN, 128, 1, 0)
  BW_CASE(true, BW_IN, 256, 0, 0)
  BW_CASE(true, BW_IN, 256, 1, 0)
  BW_CASE(false, BW_OUT, 128, 0, 0)
  BW_CASE(false, BW_OUT, 128, 1, 0)
  BW_CASE(false, BW_OUT, 256, 0, 0)
  BW_CASE(false, BW_OUT, 256, 1, 0)
  BW_CASE(true, BW_IN, 128, 0, 1)
  BW_CASE(true, BW_IN, 128, 1, 1)
  BW_CASE(true, BW_IN, 256, 0, 1)
  BW_CASE(true, BW_IN, 256, 1, 1)
  BW_CASE(false, BW_OUT, 128, 0, 1)
  BW_CASE(false, BW_OUT, 128, 1, 1)
  BW_CASE(false, BW_OUT, 256, 0, 1)
  BW_CASE(false, BW_OUT, 256, 1, 1)
#undef BW_CASE
  return CAFEQ_ERR_UNSUPPORTED;
}

// W: bf16 [d_out, d_in] with pitch ld; records and gradT as in BwParams (n_major, n_minor, NG are filled here)
static int bw_launch(cudaStream_t st, int axis_in, int k, const void* W, long long ld, BwParams p) {
  BwMaps maps;
  BwMulti mp;
  memset(&mp, 0, sizeof(mp));
  if (!make_map_bf16(&maps.w[0], W, p.d_in, p.d_out, ld, bw_box(axis_in, k))) return CAFEQ_ERR_UNSUPPORTED;
  for (int s = 1; s < BW_MAX_SUB; ++s) maps.w[s] = maps.w[0];
  mp.n = 1;
  mp.p[0] = p;
  const int swap = p.transpose_out ? 0 : 1;  // accumulator rows along the fastest index of the output
  return bw_dispatch(st, axis_in, k, swap, 0, maps, mp, g_bw_min_tiles.load(std::memory_order_relaxed));
}

// One sub-problem of a multi-matrix launch; W16 is the matrix in 16-bit storage (bf16, or the scaled fp16 copy of the
// F16 form) with pitch ld.  All sub-problems of a launch share axis, block size, output orientation and form.
struct BwSub {
  const void* W16;
  long long ld;
  BwParams p;
};

static int bw_launch_many(cudaStream_t st, int axis_in, int k, int transpose_out, int f16, const BwSub* subs, int n) {
  if (n < 1 || n > BW_MAX_SUB) return CAFEQ_ERR_INVALID_ARG;
  BwMaps maps;
  BwMulti mp;
  memset(&mp, 0, sizeof(mp));
  for (int s = 0; s < n; ++s) {
    if (!make_map_bf16(&maps.w[s], subs[s].W16, subs[s].p.d_in, subs[s].p.d_out, subs[s].ld, bw_box(axis_in, k))) return CAFEQ_ERR_UNSUPPORTED;
    mp.p[s] = subs[s].p;
    mp.p[s].transpose_out = transpose_out;
  }
  for (int s = n; s < BW_MAX_SUB; ++s) maps.w[s] = maps.w[0];
  mp.n = n;
  return bw_dispatch(st, axis_in, k, transpose_out ? 0 : 1, f16, maps, mp, 6);
}

template <int K, int SWAP_IN, int SWAP_OUT>
static int bw_launch_dual_t(cudaStream_t st, const BwMaps& mi, BwMulti pi, const BwMaps& mo, BwMulti po, bool overlap) {
  constexpr int SMEM = bw_smem<K, 1>();
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(bd_bwd_dual_kernel<K, SWAP_IN, SWAP_OUT>, SMEM, done)) return CAFEQ_ERR_CUDA;
  long long ti = 0, to = 0, maj_i = 0, maj_o = 0;
  for (int s = 0; s < pi.n; ++s) {
    bw_fill_tiles(pi.p[s], 1, K);
    ti += (long long)pi.p[s].n_major * pi.p[s].n_minor;
    maj_i += pi.p[s].n_major;
    pi.tile_end[s] = (int)ti;
  }
  for (int s = pi.n; s < BW_MAX_SUB; ++s) pi.tile_end[s] = (int)ti;
  for (int s = 0; s < po.n; ++s) {
    bw_fill_tiles(po.p[s], 0, K);
    to += (long long)po.p[s].n_major * po.p[s].n_minor;
    maj_o += po.p[s].n_major;
    po.tile_end[s] = (int)to;
  }
  for (int s = po.n; s < BW_MAX_SUB; ++s) po.tile_end[s] = (int)to;
  // tiles of the two forms hold the same bytes
  pi.stream = po.stream = l2_stream(2.0 * bw_tile(K) * K * (ti + to));
  constexpr int most = K == 256 ? 74 : 148;  // (pairs at K = 256)
  const int n_in = dual_split(ti, to, g_dual_bwd_pct.load(std::memory_order_relaxed), most);
  if (K == 256) launch_pairs_if(overlap, bd_bwd_dual_kernel<K, SWAP_IN, SWAP_OUT>, most, bw_threads<K>(), SMEM, st, mi, pi, mo, po, n_in);
  else launch_pdl_if(overlap, bd_bwd_dual_kernel<K, SWAP_IN, SWAP_OUT>, most, bw_threads<K>(), SMEM, st, mi, pi, mo, po, n_in);
  return CAFEQ_OK;
}

// fp16 single-term form only; each list holds at least 148 * 6 tiles (the caller checks with bw_dual_ok)
static bool bw_dual_ok(int k) { return k == 128 || k == 256; }
static int bw_launch_dual(cudaStream_t st, int k, int tr_in, const BwSub* in, int n_in, int tr_out, const BwSub* out, int n_out, bool overlap) {
  if (n_in < 1 || n_in > BW_MAX_SUB || n_out < 1 || n_out > BW_MAX_SUB || !bw_dual_ok(k)) return CAFEQ_ERR_INVALID_ARG;
  BwMaps mi, mo;
  BwMulti pi, po;
  memset(&pi, 0, sizeof(pi));
  memset(&po, 0, sizeof(po));
  for (int s = 0; s < n_in; ++s) {
    if (!make_map_bf16(&mi.w[s], in[s].W16, in[s].p.d_in, in[s].p.d_out, in[s].ld, bw_box(1, k))) return CAFEQ_ERR_UNSUPPORTED;
    pi.p[s] = in[s].p;
    pi.p[s].transpose_out = tr_in;
  }
  for (int s = n_in; s < BW_MAX_SUB; ++s) mi.w[s] = mi.w[0];
  for (int s = 0; s < n_out; ++s) {
    if (!make_map_bf16(&mo.w[s], out[s].W16, out[s].p.d_in, out[s].p.d_out, out[s].ld, bw_box(0, k))) return CAFEQ_ERR_UNSUPPORTED;
    po.p[s] = out[s].p;
    po.p[s].transpose_out = tr_out;
  }
  for (int s = n_out; s < BW_MAX_SUB; ++s) mo.w[s] = mo.w[0];
  pi.n = n_in;
  po.n = n_out;
  const int si = tr_in ? 0 : 1, so = tr_out ? 0 : 1;
#define BW_DUAL(KK, SI, SO) \
  if (k == KK && si == SI && so == SO) return bw_launch_dual_t<KK, SI, SO>(st, mi, pi, mo, po, overlap);
  BW_DUAL(128, 0, 0)
  BW_DUAL(128, 0, 1)
  BW_DUAL(128, 1, 0)
  BW_DUAL(128, 1, 1)
  BW_DUAL(256, 0, 0)
  BW_DUAL(256, 0, 1)
  BW_DUAL(256, 1, 0)
  BW_DUAL(256, 1, 1)
#undef BW_DUAL
  return CAFEQ_ERR_UNSUPPORTED;
}

}  // namespace cafeq
