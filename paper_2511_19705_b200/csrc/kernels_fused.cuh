// Fused block-diagonal transform pass on the 5th-generation tensor cores (sm_100a):
//   U = T o X on one axis of a bf16 matrix X, accumulated in tensor memory, followed in the same kernel by
//   the per-group work the method needs on U -- absmax / arg-max (Eq. 1's scale, Eq. 4's ||.||_inf, the
//   LogSumExp maxima), round-to-nearest codes, the residual Delta = Q(U) - U, or a sum of squares.
// U never goes to HBM.  One CTA keeps its operator block(s) resident in shared memory and streams tiles of
// X through a TMA ring; accumulators are double-buffered in tensor memory so the epilogue of tile t overlaps
// the products of tile t+1.
//
// The records of blocks of 256 run on pairs of CTAs (cta_group::2, bd_pair below): the leader issues products of 256 rows for both.
// Warp roles (576 threads): warp 0 = TMA producer, warp 1 = MMA issuer (and tensor-memory owner), warps 2..9 and 10..17 =
// two epilogue sets, one per accumulator buffer (two warps per 32-lane quarter, each owning 128 accumulator columns).
// Every wait on an mbarrier is bounded; when one runs out the kernel raises CAFEQ_ERR_TIMEOUT in the status
// word, all roles leave their loops, tensor memory is released and the kernel returns.
#pragma once

#include <atomic>
#include <mutex>
#include <type_traits>
#include <string.h>

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cafeq.h"
#include "kernels_pair_mma.cuh"

namespace cafeq {

enum { BD_IN = 0, BD_OUT = 1 };
enum { EPI_ABSMAX = 1, EPI_DELTA = 2, EPI_CODES = 4, EPI_SQSUM = 8, EPI_SURR = 16, EPI_STORE = 32 };
// compile-time kind of the epilogue: per-group records (ABSMAX, with or without SURR), records and residual, codes and
// scales only, the transformed matrix itself, its sum of squares
enum { BD_REC = 0, BD_DELTA = 1, BD_CODES = 2, BD_STORE = 3, BD_SQSUM = 4 };

struct BdParams {
  int d_out, d_in;     // shape of X
  int r;               // matrix blocks per operator block
  int t_mn;            // output axis: the operator blocks are stored transposed (T[j][i]; read as an MN-major operand)
  int pairs;           // input axis, K = 64: blocks of 32, two on the diagonal of each operator block
  int n_major;         // IN: tile columns (256 d_in columns each); OUT: row blocks (k rows each)
  int n_minor;         // IN: row tiles of 128; OUT: column tiles of NC
  int epi;
  float qmax;
  // per (row, group) records are stored GROUP-MAJOR: index = group * d_out + row
  float* a;            // [d_in / G, d_out] group absmax
  float* usel;         // signed value at the arg-max
  int* idx;            // arg-max position inside the group
  uint16_t* delta;     // bf16 [d_out, d_in], row stride d_in (EPI_STORE: U itself is written here instead of the residual)
  uint16_t* delta_lo;  // optional second bf16 term of the residual (delta + delta_lo carries 16 mantissa bits)
  int8_t* codes;       // [d_out, d_in]
  float* scales;       // [d_out, d_in / G]
  double* sqacc;
  // EPI_SURR: Eq. 4 evaluated per entry inside the pass
  const float* cw;     // input axis: sum of c_t over each column group [d_in / G]; output axis: G * c_t per row [d_out]
  float kappa;
  float* coef;         // [d_in / G, d_out] (group-major) backward coefficient 2 kappa cw a sign(U at arg-max); may be null
  double* lossacc;     // += kappa * sum cw a^2
  int a_always;        // write the maxima and their signed values even in EPI_SURR mode
  float* Aacc;         // input axis: [d_in / G] += a^2 per column group; output axis: [nbT * k] += G * sum_G a^2 per operator row
  float* vmax;         // optional: atomic maximum (bit pattern of a non-negative float) of |coef| when coefficients are
                       // written, of the group maxima otherwise
  int32_t* status;
};

// Several matrices in one launch (the problems of a layer are independent): the tiles of all sub-problems form one
// list, sub-problem s owning [tile_end[s-1], tile_end[s]), and every persistent CTA takes a contiguous run of it.
constexpr int BD_MAX_SUB = 8;
struct BdMaps {
  CUtensorMap x[BD_MAX_SUB];  // the matrices
  CUtensorMap t[BD_MAX_SUB];  // their operator blocks
};
struct BdMulti {
  int n;
  int stream;                 // read the matrices with evict_first (l2_stream below)
  int tile_end[BD_MAX_SUB];
  BdParams p[BD_MAX_SUB];     // all share one status word
};

constexpr int BD_THREADS = 64 + 2 * 256;
constexpr int BD_BOX_BYTES = 16384;  // one TMA box: 64 columns x 128 rows of bf16
// A stage is two boxes: every wait of the issuing warp costs it some 400 cycles, and the four products of one box last 512.
constexpr int BD_STAGE_BYTES = 2 * BD_BOX_BYTES;
constexpr int BD_STAGES_PER_TILE = 2;

// ------------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------------
// CTA pairs (cta_group::2): records at K = 256, where the products set the pace and a pair reads a third less of operands.  The other
// epilogues are longer than the products and lose more to a pair's larger tiles (half as many of them, of 128 KB: a last wave that is
// emptier, longer first loads) than they gain.  One CTA against pairs: codes of 4096 x 3584 17.8 us, pairs 20.1, of 14336 x 3584
// 38.9 and 40.6, of 2304 x 9216 25.1 and 29.3, residual and its square 4096 x 3584 156 and 166, apply of 2048 x 3584 13.3 and 14.0.
// Records: a 9B-shaped layer's step 343 us on pairs, 350 without, 27B-shaped with groups of 64 900 either way.
constexpr bool bd_pair(int k, int mode) { return k == 256 && mode == BD_REC; }

template <int FORM, int K, int G, int MODE>
struct BdCfg {
  // PAIR: a tile is 256 rows x 256 columns; each CTA holds half of the operator block (its 128 rows:
  // on the input axis the N half, on the output axis its accumulator rows) and half of the tile (input axis: its 128 rows; output
  // axis: its 128 columns), and its 128 rows of the accumulator.
  static constexpr bool PAIR = bd_pair(K, MODE);
  static constexpr int ROWS = PAIR ? 256 : 128;                       // IN: rows per tile
  static constexpr int NBLK = (FORM == BD_IN) ? 256 / K : 1;          // operator blocks resident per CTA
  static constexpr int T_BYTES = PAIR ? K * K : NBLK * K * K * 2;
  static constexpr int MH = (FORM == BD_OUT && !PAIR) ? K / 128 : 1;  // OUT: 128-row halves of the accumulator in this CTA
  static constexpr int NC = 256 / MH;                                 // OUT: d_in columns per tile
  static constexpr int NSTAGE = (T_BYTES > 65536) ? 3 : ((T_BYTES > 32768) ? 5 : 6);  // as many as fit
  static constexpr int SMEM = 1024 + T_BYTES + NSTAGE * BD_STAGE_BYTES + 256;
};

// The body takes the CTA's index and the number of CTAs that share its tile list, so that one launch can run two
// lists side by side (bd_pass_dual_kernel below); at K = 256 these are pairs.
template <int FORM, int K, int G, int MODE>
__device__ __forceinline__ void bd_pass_body(const BdMaps& maps, const BdMulti& mp, const int cta, const int ncta) {
  using C = BdCfg<FORM, K, G, MODE>;
  static_assert(K == 64 || K == 128 || K == 256, "block size");
  static_assert(FORM == BD_IN || K >= 128, "output-axis form needs k >= 128");
  static_assert(G == 64 || G == 128, "group size");
  constexpr bool PAIR = C::PAIR;
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  int32_t* const status = mp.p[0].status;
  const bool raised = status_raised(status);  // (awaited at the end of the set-up)

  // persistent CTA: a contiguous run of tiles in (sub-problem, major, minor) order; the operator block is reloaded
  // when the run crosses into the next major or the next sub-problem
  const int total_tiles = mp.tile_end[mp.n - 1];
  const int t_begin = (int)(((long long)cta * total_tiles) / ncta);
  const int t_end = (int)(((long long)(cta + 1) * total_tiles) / ncta);
  if (t_begin >= t_end) return;
  int s_first = 0;
  while (mp.tile_end[s_first] <= t_begin) ++s_first;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sT = smem;
  uint8_t* sStage = smem + C::T_BYTES;
  uint64_t* bars = (uint64_t*)(sStage + C::NSTAGE * BD_STAGE_BYTES);
  // barrier slots: full[NSTAGE], empty[NSTAGE], tfull[4] (one per 64-column chunk of the operator: the products on the
  // first stage of a new block start when a quarter of it has arrived), accf[2], acce[2], tfree
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8 * C::NSTAGE;
  const uint32_t bar_tfull = bar_empty + 8 * C::NSTAGE;
  const uint32_t bar_accf = bar_tfull + 32;
  const uint32_t bar_acce = bar_accf + 16;
  const uint32_t bar_tfree = bar_acce + 16;
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * C::NSTAGE + 9);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&maps.x[s_first]);
    tma_prefetch_desc(&maps.t[s_first]);
    for (int s = 0; s < C::NSTAGE; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int c = 0; c < 4; ++c) mbar_init(bar_tfull + 8 * c, 1);
    mbar_init(bar_tfree, 1);
    mbar_init(bar_accf, 1);
    mbar_init(bar_accf + 8, 1);
    mbar_init(bar_acce, PAIR ? 16 : 8);
    mbar_init(bar_acce + 8, PAIR ? 16 : 8);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      tmem_alloc_pair(smem_u32(tmem_slot), 512u);
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  bool stopped;
  if constexpr (PAIR) stopped = pair_stopped(raised, tmem_slot + 2);
  else stopped = __syncthreads_or(raised) != 0;
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  auto free_tmem = [&]() {
    if constexpr (PAIR) tmem_free_pair(tmem_base, 512u);
    else tmem_free(tmem_base, 512u);
  };
  if (stopped) {
    if (warp == 1) free_tmem();
    return;
  }

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      uint32_t it = 0, tloads = 0;
      bool ok = true;
      const uint64_t pol = l2_evict_first_policy();
      // (the leader's barriers count the loads of both CTAs)
      auto arm = [&](uint32_t bar, uint32_t bytes) {
        if constexpr (PAIR) {
          if (rank == 0) mbar_expect_tx(bar, 2 * bytes);
        } else {
          mbar_expect_tx(bar, bytes);
        }
      };
      auto load = [&](uint32_t dst, const CUtensorMap* m, int x, int y, uint32_t bar, bool hint) {
        if constexpr (PAIR) {
          if (hint) tma_load_pair_hint(dst, m, x, y, cluster_addr(bar, 0), pol);
          else tma_load_pair(dst, m, x, y, cluster_addr(bar, 0));
        } else {
          if (hint) tma_load_2d_hint(dst, m, x, y, bar, pol);
          else tma_load_2d(dst, m, x, y, bar);
        }
      };
      for (int sub = s_first; sub < mp.n && ok; ++sub) {
        const int base = sub ? mp.tile_end[sub - 1] : 0;
        if (base >= t_end) break;
        const BdParams& p = mp.p[sub];
        const CUtensorMap* tmX = &maps.x[sub];
        const CUtensorMap* tmT = &maps.t[sub];
        const int lo = (t_begin > base ? t_begin : base) - base;
        const int hi = (t_end < mp.tile_end[sub] ? t_end : mp.tile_end[sub]) - base;
        int cur_major = -1;
        for (int tile = lo; tile < hi && ok; ++tile) {
          const int major = tile / p.n_minor, t = tile - major * p.n_minor;
          if (major != cur_major) {
            // the products of the previous operator block must have finished reading it
            if (tloads > 0 && !mbar_wait(bar_tfree, (tloads - 1) & 1u, abort_flag, status)) { ok = false; break; }
            constexpr int TR = PAIR ? 128 : K;  // operator rows (columns, stored transposed) of this CTA
            for (int bi = 0; bi < C::NBLK; ++bi) {
              const int tb = (FORM == BD_IN) ? (major * C::NBLK + bi) / p.r : major / p.r;
              for (int ci = 0; ci < K / 64; ++ci) {
                const uint32_t bq = bar_tfull + 8 * (bi * (K / 64) + ci);  // at most four chunks: NBLK * K = 256 or NBLK = 1
                arm(bq, TR * 128);
                const uint32_t dst = smem_u32(sT + bi * TR * K * 2 + ci * TR * 128);
                if (FORM == BD_OUT && p.t_mn) {
                  // 64 contraction rows x TR columns as boxes of 64 x 64 (one swizzle atom each)
                  for (int j = 0; j < TR / 64; ++j) load(dst + j * 8192, tmT, (int)rank * 128 + j * 64, tb * K + ci * 64, bq, false);
                } else {
                  load(dst, tmT, ci * 64, tb * K + (int)rank * 128, bq, false);
                }
              }
            }
            cur_major = major;
            ++tloads;
          }
          for (int sidx = 0; sidx < BD_STAGES_PER_TILE; ++sidx, ++it) {
            const uint32_t s = it % C::NSTAGE, ph = (it / C::NSTAGE) & 1u;
            if (!mbar_wait(bar_empty + 8 * s, ph ^ 1u, abort_flag, status)) { ok = false; break; }
            arm(bar_full + 8 * s, BD_STAGE_BYTES);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int bx = 2 * sidx + h;
              int x, y;
              if constexpr (FORM == BD_IN) {
                x = major * 256 + bx * 64;
                y = t * C::ROWS + (int)rank * 128;
              } else if constexpr (K == 256) {  // stage = 128 contraction rows x this CTA's 128 columns
                x = t * C::NC + (int)rank * 128 + h * 64;
                y = major * K + sidx * 128;
              } else {
                x = t * C::NC + bx * 64;
                y = major * K;
              }
              load(smem_u32(sStage + s * BD_STAGE_BYTES + h * BD_BOX_BYTES), tmX, x, y, bar_full + 8 * s, mp.stream != 0);
            }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    // The whole warp runs the loop and one elected lane issues (operands in uniform registers, descriptors stepped by one
    // 32-bit addition): beside the epilogue warps a single lane that builds 64-bit descriptors took 240 cycles per
    // instruction against the 128 that a 128 x 256 x 16 product lasts.
    if (rank == 0) {  // (of a pair, the leader)
      bool ok = true;
      auto commit = [&](uint32_t bar) {
        if constexpr (PAIR) tc_commit_pair(bar);
        else tc_commit(bar);
      };
      uint32_t tfulls = 0;
      constexpr int MR = PAIR ? 256 : 128;  // accumulator rows of a product
      constexpr uint32_t idesc_in = umma_idesc_bf16(MR, K, 0, 0);
      const uint32_t sSt_u = smem_u32(sStage);
      const uint32_t tlo = umma_desc_lo(smem_u32(sT));
      uint32_t st = 0, sph = 0, tl = 0;  // stage, its phase, tile
      auto next = [&]() { if (++st == C::NSTAGE) { st = 0; sph ^= 1u; } };
      auto wait_all = [&](uint32_t bar, uint32_t ph) { return __all_sync(0xffffffffu, mbar_wait(bar, ph, abort_flag, status)) != 0; };
      for (int sub = s_first; sub < mp.n && ok; ++sub) {
        const int base = sub ? mp.tile_end[sub - 1] : 0;
        if (base >= t_end) break;
        const int n_minor = mp.p[sub].n_minor;
        const bool t_mn = FORM == BD_OUT && mp.p[sub].t_mn;
        const bool pairs = FORM == BD_IN && K == 64 && mp.p[sub].pairs;
        constexpr int NO = PAIR ? 256 : 128;
        const uint32_t idesc_out = t_mn ? umma_idesc_bf16(MR, NO, 1, 1) : umma_idesc_bf16(MR, NO, 0, 1);
        const int lo = (t_begin > base ? t_begin : base) - base;
        const int hi = (t_end < mp.tile_end[sub] ? t_end : mp.tile_end[sub]) - base;
        int left = 0;  // tiles of this sub-problem left on the current operator block
        for (int tile = lo; tile < hi && ok; ++tile, ++tl) {
          const bool fresh = left == 0;  // first tile on a newly loaded operator block
          if (fresh) left = n_minor - (tile == lo ? lo % n_minor : 0);
          const uint32_t tph = tfulls & 1u;
          if (fresh) {
            if constexpr (FORM == BD_OUT) {
              for (int c = 0; c < K / 64 && ok; ++c) ok = wait_all(bar_tfull + 8 * c, tph);
              if (!ok) break;
            }
            ++tfulls;
          }
          const uint32_t buf = tl & 1u, aph = (tl >> 1) & 1u;
          ok = wait_all(bar_acce + 8 * buf, aph ^ 1u);
          if (!ok) break;
          tc_fence_after();
          const uint32_t dbase = tmem_base + buf * 256u;
          if constexpr (FORM == BD_IN) {
#pragma unroll
            for (int sidx = 0; sidx < BD_STAGES_PER_TILE; ++sidx) {
              ok = wait_all(bar_full + 8 * st, sph);
              // box bx multiplies the operator's chunk bx
              if (ok && fresh) ok = wait_all(bar_tfull + 16 * sidx, tph) && wait_all(bar_tfull + 16 * sidx + 8, tph);
              if (!ok) break;
              tc_fence_after();
              if (elect_one()) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  const int bx = 2 * sidx + h, bi = (bx * 64) / K, ci = ((bx * 64) % K) / 64;
                  const uint32_t alo = umma_desc_lo(sSt_u + st * BD_STAGE_BYTES + h * BD_BOX_BYTES);
                  const uint32_t blo = tlo + (PAIR ? bx * 1024 : ((bi * K * K * 2 + ci * K * 128) >> 4));
                  if constexpr (PAIR) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) tc_mma_pair(dbase, alo + 2 * kk, blo + 2 * kk, idesc_in, (bx | kk) != 0 ? 1u : 0u);
                  } else if (K == 64 && pairs) {
                    // Each 32 columns meet their own block only, the diagonal quarter of the operator tile (rows 32 half ..).  The
                    // whole tile would add products with zeros: exact, but an infinity or NaN times zero is NaN.
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                      tc_mma_lo(dbase + bi * K + (kk >> 1) * 32, alo + 2 * kk, blo + (kk >> 1) * 256 + 2 * kk, umma_idesc_bf16(128, 32, 0, 0), kk & 1);
                  } else {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) tc_mma_lo(dbase + bi * K, alo + 2 * kk, blo + 2 * kk, idesc_in, (ci | kk) != 0 ? 1u : 0u);
                  }
                }
                commit(bar_empty + 8 * st);
                if (sidx == BD_STAGES_PER_TILE - 1) commit(bar_accf + 8 * buf);
              }
              __syncwarp();
              next();
            }
          } else {
            // a stage = two 64-column chunks of the same 128 weight rows: one product of N = 128 (of a pair, each CTA's half of
            // N = 256), the second swizzle atom of the MN-major operand one box further on
#pragma unroll
            for (int sidx = 0; sidx < BD_STAGES_PER_TILE; ++sidx) {
              ok = wait_all(bar_full + 8 * st, sph);
              if (!ok) break;
              tc_fence_after();
              if (elect_one()) {
                const uint32_t blo = umma_desc_lo(sSt_u + st * BD_STAGE_BYTES, BD_BOX_BYTES);
                // K-major operator: steps of 32 bytes inside the swizzled rows; MN-major: steps of sixteen 128-byte rows
                const uint32_t alo = t_mn ? umma_desc_lo(smem_u32(sT), 8192) : tlo;
                const uint32_t astep = t_mn ? 128 : 2;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                  if constexpr (PAIR)
                    tc_mma_pair(dbase, alo + (2 * sidx + ks / 4) * 1024 + (ks % 4) * astep, blo + ks * 128, idesc_out, (sidx | ks) != 0 ? 1u : 0u);
                  else if constexpr (K == 256)  // both halves of the operator's rows against the same columns
#pragma unroll
                    for (int mh = 0; mh < 2; ++mh)
                      tc_mma_lo(dbase + mh * 128, alo + (2 * sidx + ks / 4) * 2048 + mh * 1024 + (ks % 4) * astep, blo + ks * 128, idesc_out,
                                (sidx | ks) != 0 ? 1u : 0u);
                  else
                    tc_mma_lo(dbase + sidx * 128, alo + (ks / 4) * 1024 + (ks % 4) * astep, blo + ks * 128, idesc_out, ks != 0 ? 1u : 0u);
                }
                commit(bar_empty + 8 * st);
                if (sidx == BD_STAGES_PER_TILE - 1) commit(bar_accf + 8 * buf);
              }
              __syncwarp();
              next();
            }
          }
          // last tile of this operator block with more to come: signal when its products are done with the block
          if (--left == 0 || tile + 1 == hi) {
            if (ok && base + tile + 1 < t_end && elect_one()) commit(bar_tfree);
            __syncwarp();
          }
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    // Set `buf` (eight warps) serves the tiles of accumulator buffer `buf`, so a tile's epilogue may last as long as two
    // tiles' products.  With one set of eight warps for both buffers the epilogue was the longest stage: its dependent
    // chains left the issue slots of two warps per scheduler mostly empty (records 3200 cycles a tile, codes 10400,
    // against 2100 for the products and 2800 for the bytes).  Measured, one set -> two: records of a 9B-shaped layer (both
    // forms, 198 M weights) 127 -> 111 us, 27B-shaped with groups of 64 (515 M) 325 -> 286; codes of 14336 x 3584 86 -> 50;
    // the transformed matrix of 8192 x 2304 29.5 -> 20.5 (with its stores widened to whole sectors).
    // Since then, records of the same layer, back to back: 105 us; arg-max by chunks and loads in flight 95 (without an epilogue 86,
    // without loads 94, with a quarter of the products 94), stages of two boxes 93, blocks of 256 on CTA pairs 89.  There the
    // products (2048 cycles a tile at K = 256) take 84 % of a CTA's time, at the clock that the power limit leaves.
    const int q = warp & 3, hw = ((warp - 2) >> 2) & 1;
    const uint32_t buf = (uint32_t)((warp - 2) >> 3);
    const int L = q * 32 + lane;
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + buf * 256u + hw * 128u;
    uint32_t tl = 0, aph = 0;
    bool ok = true;
    constexpr int NG = 128 / G;
    for (int sub = s_first; sub < mp.n && ok; ++sub) {
      const int base = sub ? mp.tile_end[sub - 1] : 0;
      if (base >= t_end) break;
      const BdParams& p = mp.p[sub];
      const int lo = (t_begin > base ? t_begin : base) - base;
      const int hi = (t_end < mp.tile_end[sub] ? t_end : mp.tile_end[sub]) - base;
      const int n_minor = p.n_minor;
      int major = lo / n_minor, t = lo - major * n_minor - 1;
      double sq_local = 0.0, sur_local = 0.0;
      float asum[NG], vm = 0.f;  // Eq. 4: squared maxima summed over the tiles of one block (input axis: per column group;
      int asum_key = -1;         // output axis: per row, in asum[0]), and which block / row they belong to
#pragma unroll
      for (int gi = 0; gi < NG; ++gi) asum[gi] = 0.f;
      bool bad = false;
      auto flush_asum = [&]() {
        if constexpr (FORM == BD_IN) {
          const int c0 = asum_key * 256 + hw * 128;
#pragma unroll
          for (int gi = 0; gi < NG; ++gi) {
            float a2 = asum[gi];
            for (int o = 16; o > 0; o >>= 1) a2 += __shfl_xor_sync(0xffffffffu, a2, o);
            if (lane == 0 && a2 != 0.f && c0 < p.d_in) atomicAdd(&p.Aacc[c0 / G + gi], a2);
            asum[gi] = 0.f;
          }
        } else {
          if (asum[0] != 0.f) {
            const int Bq = asum_key / K;
            atomicAdd(&p.Aacc[(Bq / p.r) * K + (asum_key - Bq * K)], (float)G * asum[0]);
          }
          asum[0] = 0.f;
        }
      };
      for (int tile = lo; tile < hi && ok; ++tile, ++tl) {
        if (++t == n_minor) { t = 0; ++major; }
        if ((tl & 1u) != buf) continue;
        int row, col0;
        if constexpr (FORM == BD_IN) {
          row = t * C::ROWS + (int)rank * 128 + L;
          col0 = major * 256 + hw * 128;
        } else {
          row = major * K + ((int)rank + (C::MH == 2 ? hw : 0)) * 128 + L;
          col0 = t * C::NC + (C::MH == 2 ? 0 : hw * 128);
        }
        const bool valid = (row < p.d_out) && (col0 < p.d_in);
        // Eq. 4 weights of this thread's groups, requested before the wait for the accumulator so that the
        // global-memory latency is hidden behind it
        float wgt[NG];
        if constexpr (MODE == BD_REC || MODE == BD_DELTA) {
#pragma unroll
          for (int gi = 0; gi < NG; ++gi) wgt[gi] = 0.f;
          if ((p.epi & EPI_SURR) && valid) {
#pragma unroll
            for (int gi = 0; gi < NG; ++gi) wgt[gi] = (FORM == BD_IN) ? ld_plain(p.cw + col0 / G + gi) : ld_plain(p.cw + row);
          }
        }
        ok = __all_sync(0xffffffffu, mbar_wait(bar_accf + 8 * buf, aph, abort_flag, status));
        aph ^= 1u;
        if (!ok) break;
        tc_fence_after();
        auto release = [&]() {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if constexpr (PAIR) mbar_arrive_pair_tmem(cluster_addr(bar_acce + 8 * buf, 0));
            else mbar_arrive(bar_acce + 8 * buf);
          }
        };
        // This thread's columns from `addr` on, N times 16, the next 16 requested while these are worked on (unrolled: a copy of the
        // registers in flight would read them too early).
        auto walk = [&](uint32_t addr, auto count, auto&& f) {
          constexpr int N = decltype(count)::value;
          uint32_t raw[2][16];
          tc_ld16_async(addr, raw[0]);
#pragma unroll
          for (int ch = 0; ch < N; ++ch) {
            tc_ld16_wait(raw[ch & 1]);
            if (ch < N - 1) tc_ld16_async(addr + (ch + 1) * 16, raw[(ch + 1) & 1]);
            float v[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = __uint_as_float(raw[ch & 1][e]);
            f(ch, v);
          }
        };
        constexpr std::integral_constant<int, 8> all{};        // its 128 columns
        constexpr std::integral_constant<int, G / 16> group{};  // those of a group
        if constexpr (MODE == BD_STORE) {
          // the transformed matrix itself, rounded to bf16 (inference-side apply of a block-diagonal operator)
          uint16_t* dst = p.delta + (long long)row * p.d_in + col0;
          const bool wide = ((uintptr_t)p.delta & 31) == 0;
          walk(taddr, all, [&](int ch, const float* v) {
            if (ch == 7) release();
            uint32_t pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2)
              pk[e >> 1] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[e])) |
                           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[e + 1])) << 16);
            if (valid) store32(dst + ch * 16, pk, wide);
          });
        } else if constexpr (MODE == BD_SQSUM) {
          // sum of squares only (second pass of the l2 proxy)
          float sq4[4] = {0.f, 0.f, 0.f, 0.f};
          walk(taddr, all, [&](int ch, const float* v) {
            if (ch == 7) release();
#pragma unroll
            for (int e = 0; e < 16; ++e) sq4[e & 3] = fmaf(v[e], v[e], sq4[e & 3]);
          });
          sq_local += valid ? (double)((sq4[0] + sq4[1]) + (sq4[2] + sq4[3])) : 0.0;
        } else if constexpr (MODE == BD_CODES) {
          // Group after group (both groups of 64 at once took more registers than there are: 14336 x 3584 at k = 128 40.5 -> 43 us).
          //
          // code = rne(fl32(u / s)).  The IEEE division is a long dependent sequence with a slow-path branch per
          // element; u * (1 / s), rounded once together with its addend below, differs from fl32(u / s) by less than
          // (qmax + 1) * 2.4e-7, so it rounds to the same integer unless the quotient lies within that distance of a
          // half-integer: those (rare: the transformed values are not on a coarse grid) chunks are redone with the
          // division.  The rounding uses no conversion instruction: t = u / s + 1.5 * 2^23 holds rne(u / s) in its low
          // mantissa bits (an fp32 result rounds to nearest even, as rintf does) and, 0x4B400000 having a zero low
          // byte, the low byte of t's pattern is the two's-complement code; |u / s| <= qmax (1 + 3 * 2^-23), so
          // nothing is clamped.
          constexpr float MAGIC = 12582912.f;
          const float win = 0.5f - (p.qmax + 1.f) * 1.0e-6f;
          const bool wide = ((uintptr_t)p.codes & 31) == 0;
#pragma unroll 1
          for (int gi = 0; gi < NG; ++gi) {
            const uint32_t gaddr = taddr + gi * G;
            // the absmax: two columns per instruction, NaN and infinity stay visible in the maximum
            float m2[2] = {0.f, 0.f};
            walk(gaddr, group, [&](int, const float* v) {
#pragma unroll
              for (int e = 0; e < 16; e += 2) m2[(e >> 1) & 1] = max_abs2(m2[(e >> 1) & 1], v[e], v[e + 1]);
            });
            float best = max_abs2(m2[0], m2[1], 0.f);
            if (valid && !(best <= 3.0e38f)) bad = true;
            // A group with a NaN keeps the maximum of its numbers (a non-finite weight spoils its own block only; the NaN itself
            // is coded -qmax): one more walk, by the whole warp, where any lane has met one.
            if (__any_sync(0xffffffffu, best != best)) {
              best = 0.f;
#pragma unroll 1
              for (int ch = 0; ch < G / 16; ++ch) {
                float v[16];
                tc_ld16(gaddr + ch * 16, v);
#pragma unroll
                for (int e = 0; e < 16; ++e) best = fmaxf(best, fabsf(v[e]));
              }
            }
            const float s = __fdiv_rn(best, p.qmax);
            const float rs = (s > 0.f) ? __frcp_rn(s) : 0.f;
            if (valid) p.scales[(long long)row * (p.d_in / G) + (col0 / G + gi)] = s;
            int8_t* dst = p.codes + (long long)row * p.d_in + col0 + gi * G;
            uint32_t cpk[8];
            float dm = 0.f;
            walk(gaddr, group, [&](int hc, const float* v) {
              const int ch = hc >> 1, hf = hc & 1;  // 32 columns a store
              if (hf == 0) dm = 0.f;
#pragma unroll
              for (int w = 0; w < 4; ++w) {
                uint32_t cb[4];
                float d[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const float x = v[4 * w + e];
                  const float tt = fmaf(x, rs, MAGIC);
                  cb[e] = __float_as_uint(tt);
                  d[e] = fmaf(x, rs, -(tt - MAGIC));
                }
                dm = max_abs2(dm, d[0], d[1]);
                dm = max_abs2(dm, d[2], d[3]);
                cpk[4 * hf + w] = __byte_perm(__byte_perm(cb[0], cb[1], 0x0040), __byte_perm(cb[2], cb[3], 0x0040), 0x5410);
              }
              if (hf == 0) return;
              // (also: a scale so small that its reciprocal overflows); the accumulator is read again by the whole warp
              if (__any_sync(0xffffffffu, !(dm <= win) || !(rs < 3.0e38f))) {
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                  float u[16];
                  tc_ld16(gaddr + ch * 32 + h2 * 16, u);
#pragma unroll
                  for (int w = 0; w < 4; ++w) {
                    uint32_t pk = 0;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                      float qd = (s > 0.f) ? rintf(__fdiv_rn(u[4 * w + e], s)) : 0.f;
                      qd = fminf(fmaxf(qd, -p.qmax), p.qmax);
                      pk |= ((uint32_t)((int)qd) & 0xFFu) << (8 * e);
                    }
                    cpk[4 * h2 + w] = pk;
                  }
                }
              }
              if (ch == G / 32 - 1 && gi == NG - 1) release();
              if (valid) store32(dst + ch * 32, cpk, wide);
            });
          }
        } else {
          float best[NG], bval[NG];
          int bidx[NG];
#pragma unroll
          for (int gi = 0; gi < NG; ++gi) { best[gi] = 0.f; bval[gi] = 0.f; bidx[gi] = 0; }
          // Group absmax with arg-max.  Per chunk of 16 columns the maximum (two columns per instruction), and where it beats the
          // chunks before it the chunk itself is kept, one select per column; the position inside the kept chunk is looked up
          // once per group.  1.7 instructions per column and no long chains (compare, two selects and the range check per
          // column took 4, in four chains), the next chunk's loads in flight meanwhile.  A strict comparison keeps the lowest
          // of equal chunks, the downward search the lowest column.
          float kept[16], nm = 0.f;
          int kc = 0;
          float b = 0.f;
#pragma unroll
          for (int e = 0; e < 16; ++e) kept[e] = 0.f;
          walk(taddr, all, [&](int ch, const float* r) {
            constexpr int CPG = G / 16;  // chunks per group
            const int gi = ch / CPG;
            float m[2] = {0.f, 0.f};
#pragma unroll
            for (int e = 0; e < 16; e += 2) m[(e >> 1) & 1] = max_abs2(m[(e >> 1) & 1], r[e], r[e + 1]);
            const float cm = max_abs2(m[0], m[1], 0.f);
            nm = max_abs2(nm, cm, 0.f);
            const bool up = cm > b;
            b = up ? cm : b;
            kc = up ? ch % CPG : kc;
#pragma unroll
            for (int e = 0; e < 16; ++e) kept[e] = up ? r[e] : kept[e];
            if (ch % CPG == CPG - 1) {
              float v = 0.f;
              int ix = 0;
#pragma unroll
              for (int e = 15; e >= 0; --e)
                if (fabsf(kept[e]) == b) { v = kept[e]; ix = e; }
              best[gi] = b;
              bval[gi] = v;
              bidx[gi] = kc * 16 + ix;
              b = 0.f;
              kc = 0;
#pragma unroll
              for (int e = 0; e < 16; ++e) kept[e] = 0.f;
            }
          });
          if (__any_sync(0xffffffffu, nm != nm)) {
            // A NaN hides its chunk from the comparisons above: the groups' maxima over their numbers, by the whole warp.
#pragma unroll
            for (int gi = 0; gi < NG; ++gi) {
              best[gi] = bval[gi] = 0.f;
              bidx[gi] = 0;
#pragma unroll 1
              for (int ch = 0; ch < G / 16; ++ch) {
                float v[16];
                tc_ld16(taddr + gi * G + ch * 16, v);
#pragma unroll
                for (int e = 0; e < 16; ++e)
                  if (fabsf(v[e]) > best[gi]) { best[gi] = fabsf(v[e]); bval[gi] = v[e]; bidx[gi] = ch * 16 + e; }
              }
            }
          }
          if (valid && !(nm <= 3.0e38f)) bad = true;
          // Without a second walk over the accumulator (codes / residual) everything still needed is in registers:
          // hand the buffer back to the tensor cores now.  The arrive has release semantics, so issuing it after the
          // global stores below would make every tile wait for those stores to land.
          if constexpr (MODE == BD_REC) release();
          if (valid && p.vmax && !((p.epi & EPI_SURR) && p.coef)) {
#pragma unroll
            for (int gi = 0; gi < NG; ++gi) vm = fmaxf(vm, best[gi]);
          }
          if (valid) {
            // with Eq. 4 evaluated right here nothing downstream reads the maxima or their signs: the backward only
            // needs (arg-max index, coefficient).  Every scattered 4-byte store is a partial-sector write at L2.
            const bool need_a = !(p.epi & EPI_SURR) || p.a_always;
#pragma unroll
            for (int gi = 0; gi < NG; ++gi) {
              // group-major records: consecutive rows of one group are contiguous, so a warp's store is one line
              const long long w = (long long)(col0 / G + gi) * p.d_out + row;
              if (need_a) {
                p.a[w] = best[gi];
                p.usel[w] = bval[gi];
              }
              p.idx[w] = bidx[gi];
            }
          }
          if (p.epi & EPI_SURR) {
            const int key = (FORM == BD_IN) ? major : row;  // (uniform over the warp on the input axis)
            if (asum_key != key) {
              if (asum_key >= 0) flush_asum();
              asum_key = key;
            }
            float surf = 0.f;
#pragma unroll
            for (int gi = 0; gi < NG; ++gi) {
              const float av = valid ? best[gi] : 0.f;
              surf = fmaf(wgt[gi] * av, av, surf);
              if (valid && p.coef) {
                const float sg = (bval[gi] > 0.f) ? 1.f : ((bval[gi] < 0.f) ? -1.f : 0.f);
                const float cf = 2.f * p.kappa * wgt[gi] * av;
                p.coef[(long long)(col0 / G + gi) * p.d_out + row] = cf * sg;
                vm = fmaxf(vm, cf);
              }
              float& as = asum[(FORM == BD_IN) ? gi : 0];
              as = fmaf(av, av, as);
            }
            sur_local += (double)surf;
          }
          if constexpr (MODE == BD_DELTA) {
            // residual s * code - u as one or two bf16 terms, 16 columns at a time (rounding as above)
            constexpr float MAGIC = 12582912.f;
            const float win = 0.5f - (p.qmax + 1.f) * 1.0e-6f;
            uint16_t* dst = p.delta + (long long)row * p.d_in + col0;
            uint16_t* dst_lo = p.delta_lo ? p.delta_lo + (long long)row * p.d_in + col0 : nullptr;
            const bool wide = (((uintptr_t)p.delta | (uintptr_t)p.delta_lo) & 31) == 0;
            auto put = [&](int ch, const float* v, const float* qv, float s) {
              uint32_t hpk[8], lpk[8];
#pragma unroll
              for (int e = 0; e < 16; e += 2) {
                const float d0 = s * qv[e] - v[e], d1 = s * qv[e + 1] - v[e + 1];
                const __nv_bfloat16 b0 = __float2bfloat16_rn(d0), b1 = __float2bfloat16_rn(d1);
                hpk[e >> 1] = (uint32_t)__bfloat16_as_ushort(b0) | ((uint32_t)__bfloat16_as_ushort(b1) << 16);
                lpk[e >> 1] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(d0 - __bfloat162float(b0))) |
                              ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(d1 - __bfloat162float(b1))) << 16);
              }
              if (valid) {
                store32(dst + ch * 16, hpk, wide);
                if (dst_lo) store32(dst_lo + ch * 16, lpk, wide);
              }
            };
            float s[NG], rs[NG];
            uint32_t redo = 0;
#pragma unroll
            for (int gi = 0; gi < NG; ++gi) {
              s[gi] = __fdiv_rn(best[gi], p.qmax);
              rs[gi] = (s[gi] > 0.f) ? __frcp_rn(s[gi]) : 0.f;
            }
            auto put16 = [&](int ch, const float* v, float sg, float r) {
              float dm = 0.f, qv[16];
#pragma unroll
              for (int e = 0; e < 16; e += 2) {
                qv[e] = fmaf(v[e], r, MAGIC) - MAGIC;
                qv[e + 1] = fmaf(v[e + 1], r, MAGIC) - MAGIC;
                dm = max_abs2(dm, fmaf(v[e], r, -qv[e]), fmaf(v[e + 1], r, -qv[e + 1]));
              }
              if (__any_sync(0xffffffffu, !(dm <= win) || !(r < 3.0e38f))) redo |= 1u << ch;
              if (ch == 7 && !redo) release();
              put(ch, v, qv, sg);
            };
            // (rolled: unrolled, with the next columns in flight, the code is eight times as long; Eq. 3's loss of 4096 x 3584 at k = 256
            // 162 us, after other work 174, so 156 and 164)
#pragma unroll 1
            for (int ch = 0; ch < 8; ++ch) {
              float v[16];
              tc_ld16(taddr + ch * 16, v);
              put16(ch, v, (NG == 1 || ch < 4) ? s[0] : s[NG - 1], (NG == 1 || ch < 4) ? rs[0] : rs[NG - 1]);
            }
            if (redo) {
#pragma unroll 1
              for (int ch = 0; ch < 8; ++ch) {
                if (!((redo >> ch) & 1u)) continue;
                const float s1 = (NG == 1 || ch < 4) ? s[0] : s[NG - 1];
                float u[16], qv[16];
                tc_ld16(taddr + ch * 16, u);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                  const float qd = (s1 > 0.f) ? rintf(__fdiv_rn(u[e], s1)) : 0.f;
                  qv[e] = fminf(fmaxf(qd, -p.qmax), p.qmax);
                }
                put(ch, u, qv, s1);
              }
              release();
            }
          }
        }
      }
      if constexpr (MODE == BD_SQSUM) {
        for (int o = 16; o > 0; o >>= 1) sq_local += __shfl_xor_sync(0xffffffffu, sq_local, o);
        if (lane == 0 && sq_local != 0.0) atomicAdd(p.sqacc, sq_local);
      }
      if constexpr (MODE == BD_REC || MODE == BD_DELTA) {
        if (p.epi & EPI_SURR) {
          for (int o = 16; o > 0; o >>= 1) sur_local += __shfl_xor_sync(0xffffffffu, sur_local, o);
          if (lane == 0 && sur_local != 0.0) atomicAdd(p.lossacc, (double)p.kappa * sur_local);
          if (asum_key >= 0) flush_asum();
        }
        if (p.vmax) {
          for (int o = 16; o > 0; o >>= 1) vm = fmaxf(vm, __shfl_xor_sync(0xffffffffu, vm, o));
          if (lane == 0 && vm > 0.f) atomicMax(reinterpret_cast<int*>(p.vmax), __float_as_int(vm));
        }
      }
      if (__any_sync(0xffffffffu, bad) && lane == 0) raise_status(status, CAFEQ_ERR_NONFINITE);
    }  // sub-problems
  }

  // ---------------------------------------------------------------- teardown
  pdl_release();
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // (neither CTA leaves while the other's products may read its shared memory)
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    free_tmem();
  }
}

template <int FORM, int K, int G, int MODE>
__global__ void __launch_bounds__(BD_THREADS, 1)
bd_pass_kernel(const __grid_constant__ BdMaps maps, const __grid_constant__ BdMulti mp) {
  pdl_wait();
  constexpr int W = BdCfg<FORM, K, G, MODE>::PAIR ? 2 : 1;
  bd_pass_body<FORM, K, G, MODE>(maps, mp, (int)blockIdx.x / W, (int)gridDim.x / W);
}

// Both forms in one launch: the first n_in CTAs run the input-axis list, the others the output-axis list (a layer
// has matrices of both forms; two launches pay the fixed cost of a persistent kernel -- operator load, pipeline
// fill, the tail of the slowest CTA -- twice, and the smaller list alone cannot fill the memory system).
template <int K, int G>
__global__ void __launch_bounds__(BD_THREADS, 1)
bd_pass_dual_kernel(const __grid_constant__ BdMaps maps_in, const __grid_constant__ BdMulti mp_in,
                    const __grid_constant__ BdMaps maps_out, const __grid_constant__ BdMulti mp_out, const int n_in) {
  pdl_wait();
  constexpr int W = BdCfg<BD_IN, K, G, BD_REC>::PAIR ? 2 : 1;
  const int cta = (int)blockIdx.x / W, n = (int)gridDim.x / W;  // (pairs at K = 256)
  if (cta < n_in) bd_pass_body<BD_IN, K, G, BD_REC>(maps_in, mp_in, cta, n_in);
  else bd_pass_body<BD_OUT, K, G, BD_REC>(maps_out, mp_out, cta - n_in, n - n_in);
}

// ------------------------------------------------------------------------------------------------
// host side: tensor maps and launch
// ------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)ptr;
  });
  return fn;
}

// 2-D bf16 tensor map: `cols` contiguous elements per row, `rows` rows, row pitch in elements, box 64 x box_rows,
// 128-byte swizzle, out-of-range elements read as zero.
static bool make_map_bf16(CUtensorMap* m, const void* base, long long cols, long long rows, long long pitch, int box_rows) {
  EncodeTiledFn enc = get_encode_tiled();
  if (!enc) return false;
  if (((uintptr_t)base & 15) || ((pitch * 2) & 15)) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)pitch * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Shapes the fused pass covers; everything else runs on the shape-agnostic kernels.
static bool bd_supported(int form, int d_out, int d_in, long long ld, int k, int g, const void* X) {
  if (!(g == 64 || g == 128)) return false;
  if (form == BD_IN) {
    if (!(k == 64 || k == 128 || k == 256)) return false;
    if (d_in % 128) return false;  // (a half tile past the end reads zeros and stores nothing)
  } else {
    if (!(k == 128 || k == 256)) return false;
    if (d_out % k || d_in % 128) return false;
  }
  if ((ld % 8) || ((uintptr_t)X & 15)) return false;
  return true;
}

// Weights of a launch that take more than a quarter of L2 (126 MB) are read with evict_first, so that they displace one
// another and not what the step comes back to (records, operators, k x k state).  Measured: layer step of a 2B-shaped pair
// (85 MB) 148 -> 139 us, of a 42 MB pair 115 -> 107, of a 9B-shaped layer 410 -> 399; codes of 103 MB 72 -> 69; layers of
// 6 to 20 MB the same either way.  Not for the inference side: activations usually come from the product before, through
// L2 (38 MB read again and again: 23.6 us, with the hint 25.7).
static int l2_stream(double bytes) { return bytes > 32.0 * (1 << 20) ? 1 : 0; }

static std::atomic<int> g_bd_min_tiles{1};

// opt the kernel into its dynamic shared memory once per device (the attribute is per device and per function)
template <typename KernelT>
static bool opt_in_smem(KernelT kernel, int bytes, std::atomic<unsigned long long>& done_mask) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done_mask.load(std::memory_order_acquire) & bit) return true;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
  done_mask.fetch_or(bit, std::memory_order_release);
  return true;
}

// tile geometry of one sub-problem
template <int FORM, int K, int G, int MODE>
static void bd_fill_tiles(BdParams& p) {
  using C = BdCfg<FORM, K, G, MODE>;
  if (FORM == BD_IN) {
    p.n_major = (p.d_in + 255) / 256;
    p.n_minor = (p.d_out + C::ROWS - 1) / C::ROWS;
  } else {
    p.n_major = p.d_out / K;
    p.n_minor = (p.d_in + C::NC - 1) / C::NC;
  }
}

template <int FORM, int K, int G, int MODE>
static int bd_launch_multi_t(cudaStream_t st, const BdMaps& maps, BdMulti mp, int min_tiles) {
  using C = BdCfg<FORM, K, G, MODE>;
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(bd_pass_kernel<FORM, K, G, MODE>, C::SMEM, done)) return CAFEQ_ERR_CUDA;
  long long total = 0;
  for (int s = 0; s < mp.n; ++s) {
    bd_fill_tiles<FORM, K, G, MODE>(mp.p[s]);
    total += (long long)mp.p[s].n_major * mp.p[s].n_minor;
    mp.tile_end[s] = (int)total;
  }
  for (int s = mp.n; s < BD_MAX_SUB; ++s) mp.tile_end[s] = (int)total;
  mp.stream = (MODE == BD_REC || MODE == BD_CODES) ? l2_stream(512.0 * C::ROWS * total) : 0;
  // one persistent CTA per SM at most; when several problems overlap in streams, small matrices take fewer CTAs
  // (at least min_tiles tiles each): the fixed cost of a CTA is spread over more tiles and the SMs left over
  // run another problem's kernel
  long long want = total / (min_tiles > 0 ? min_tiles : 1);
  if (want < 1) want = 1;
  constexpr int most = C::PAIR ? 74 : 148;
  const int grid = want < most ? (int)want : most;
  if (C::PAIR) launch_pairs_if(true, bd_pass_kernel<FORM, K, G, MODE>, grid, BD_THREADS, C::SMEM, st, maps, mp);
  else launch_pdl(bd_pass_kernel<FORM, K, G, MODE>, grid, BD_THREADS, C::SMEM, st, maps, mp);
  return CAFEQ_OK;
}

// the sub-problems of a launch share the kind of their epilogue
static int bd_mode(int epi) {
  if (epi & EPI_STORE) return BD_STORE;
  if (epi & EPI_SQSUM) return BD_SQSUM;
  if (epi & EPI_CODES) return BD_CODES;
  return (epi & EPI_DELTA) ? BD_DELTA : BD_REC;
}

// rows of the operator in one box: all of a block, of a pair's CTA its half; stored transposed, one swizzle atom
static int bd_operator_rows(int k, const BdParams& p) { return p.t_mn ? 64 : (bd_pair(k, bd_mode(p.epi)) ? 128 : k); }

template <int FORM, int K, int G>
static int bd_dispatch_mode(cudaStream_t st, const BdMaps& maps, const BdMulti& mp, int min_tiles) {
  switch (bd_mode(mp.p[0].epi)) {
    case BD_REC: return bd_launch_multi_t<FORM, K, G, BD_REC>(st, maps, mp, min_tiles);
    case BD_DELTA: return bd_launch_multi_t<FORM, K, G, BD_DELTA>(st, maps, mp, min_tiles);
    case BD_CODES: return bd_launch_multi_t<FORM, K, G, BD_CODES>(st, maps, mp, min_tiles);
    // (the group width plays no part in these two)
    case BD_STORE: return bd_launch_multi_t<FORM, K, 128, BD_STORE>(st, maps, mp, min_tiles);
    default: return bd_launch_multi_t<FORM, K, 128, BD_SQSUM>(st, maps, mp, min_tiles);
  }
}

static int bd_dispatch(cudaStream_t st, int form, int k, int g, const BdMaps& maps, const BdMulti& mp, int min_tiles) {
#define BD_CASE(F, KK, GG) \
  if (form == F && k == KK && g == GG) return bd_dispatch_mode<F, KK, GG>(st, maps, mp, min_tiles);
  BD_CASE(BD_IN, 64, 64)
  BD_CASE(BD_IN, 64, 128)
  BD_CASE(BD_IN, 128, 64)
  BD_CASE(BD_IN, 128, 128)
  BD_CASE(BD_IN, 256, 64)
  BD_CASE(BD_IN, 256, 128)
  BD_CASE(BD_OUT, 128, 64)
  BD_CASE(BD_OUT, 128, 128)
  BD_CASE(BD_OUT, 256, 64)
  BD_CASE(BD_OUT, 256, 128)
#undef BD_CASE
  return CAFEQ_ERR_UNSUPPORTED;
}

// X: bf16 [d_out, d_in] with pitch ld; Tb: bf16 operator blocks [nbT * k, k] in applied orientation.
static int bd_launch(cudaStream_t st, int form, int k, int g, const void* X, long long ld, const void* Tb, int nbT, BdParams p) {
  BdMaps maps;
  BdMulti mp;
  memset(&mp, 0, sizeof(mp));
  if (!make_map_bf16(&maps.x[0], X, p.d_in, p.d_out, ld, 128)) return CAFEQ_ERR_UNSUPPORTED;
  if (!make_map_bf16(&maps.t[0], Tb, k, (long long)nbT * k, k, bd_operator_rows(k, p))) return CAFEQ_ERR_UNSUPPORTED;
  for (int s = 1; s < BD_MAX_SUB; ++s) { maps.x[s] = maps.x[0]; maps.t[s] = maps.t[0]; }
  mp.n = 1;
  mp.p[0] = p;
  return bd_dispatch(st, form, k, g, maps, mp, g_bd_min_tiles.load(std::memory_order_relaxed));
}

// One sub-problem of a multi-matrix launch: the matrix, its operator blocks (bf16, applied orientation) and its
// epilogue parameters (d_out, d_in, r, epi, ... filled by the caller).
struct BdSub {
  const void* X;
  long long ld;
  const void* Tb;
  int nbT;
  BdParams p;
};

// Up to BD_MAX_SUB matrices of the same form, block size and group size in one persistent launch.
static int bd_launch_many(cudaStream_t st, int form, int k, int g, const BdSub* subs, int n) {
  if (n < 1 || n > BD_MAX_SUB) return CAFEQ_ERR_INVALID_ARG;
  BdMaps maps;
  BdMulti mp;
  memset(&mp, 0, sizeof(mp));
  for (int s = 0; s < n; ++s) {
    if (!make_map_bf16(&maps.x[s], subs[s].X, subs[s].p.d_in, subs[s].p.d_out, subs[s].ld, 128)) return CAFEQ_ERR_UNSUPPORTED;
    if (!make_map_bf16(&maps.t[s], subs[s].Tb, k, (long long)subs[s].nbT * k, k, bd_operator_rows(k, subs[s].p))) return CAFEQ_ERR_UNSUPPORTED;
    mp.p[s] = subs[s].p;
  }
  for (int s = n; s < BD_MAX_SUB; ++s) { maps.x[s] = maps.x[0]; maps.t[s] = maps.t[0]; }
  mp.n = n;
  return bd_dispatch(st, form, k, g, maps, mp, 1);
}

// relative cost of an output-axis tile against an input-axis tile of the same bytes (measured per-tile times of
// the two forms): sets how the CTAs of a dual launch are divided
static std::atomic<int> g_dual_pass_pct{110}, g_dual_bwd_pct{100};

static int dual_split(long long tiles_in, long long tiles_out, int out_weight_pct, int n = 148) {
  const double wi = (double)tiles_in, wo = (double)tiles_out * out_weight_pct / 100.0;
  int n_in = (int)(n * wi / (wi + wo) + 0.5);
  if (n_in < 1) n_in = 1;
  if (n_in > n - 1) n_in = n - 1;
  return n_in;
}

template <int K, int G>
static int bd_launch_dual_t(cudaStream_t st, const BdMaps& mi, BdMulti pi, const BdMaps& mo, BdMulti po, bool overlap) {
  constexpr int SMEM = BdCfg<BD_IN, K, G, BD_REC>::SMEM > BdCfg<BD_OUT, K, G, BD_REC>::SMEM ? BdCfg<BD_IN, K, G, BD_REC>::SMEM : BdCfg<BD_OUT, K, G, BD_REC>::SMEM;
  static std::atomic<unsigned long long> done{0};
  if (!opt_in_smem(bd_pass_dual_kernel<K, G>, SMEM, done)) return CAFEQ_ERR_CUDA;
  long long ti = 0, to = 0;
  for (int s = 0; s < pi.n; ++s) {
    bd_fill_tiles<BD_IN, K, G, BD_REC>(pi.p[s]);
    ti += (long long)pi.p[s].n_major * pi.p[s].n_minor;
    pi.tile_end[s] = (int)ti;
  }
  for (int s = pi.n; s < BD_MAX_SUB; ++s) pi.tile_end[s] = (int)ti;
  for (int s = 0; s < po.n; ++s) {
    bd_fill_tiles<BD_OUT, K, G, BD_REC>(po.p[s]);
    to += (long long)po.p[s].n_major * po.p[s].n_minor;
    po.tile_end[s] = (int)to;
  }
  for (int s = po.n; s < BD_MAX_SUB; ++s) po.tile_end[s] = (int)to;
  constexpr bool PAIR = BdCfg<BD_IN, K, G, BD_REC>::PAIR;
  pi.stream = po.stream = l2_stream((PAIR ? 131072.0 : 65536.0) * (ti + to));
  const int n_in = dual_split(ti, to, g_dual_pass_pct.load(std::memory_order_relaxed), PAIR ? 74 : 148);
  if (PAIR) launch_pairs_if(overlap, bd_pass_dual_kernel<K, G>, 74, BD_THREADS, SMEM, st, mi, pi, mo, po, n_in);
  else launch_pdl_if(overlap, bd_pass_dual_kernel<K, G>, 148, BD_THREADS, SMEM, st, mi, pi, mo, po, n_in);
  return CAFEQ_OK;
}

// Input-axis and output-axis matrices of one block size and group size in ONE persistent launch (both lists
// non-empty, each at least 148 tiles so that every CTA has work; otherwise the caller launches them separately).
static bool bd_dual_ok(int k, int g) { return (k == 128 || k == 256) && (g == 64 || g == 128); }
static int bd_launch_dual(cudaStream_t st, int k, int g, const BdSub* in, int n_in, const BdSub* out, int n_out, bool overlap) {
  if (n_in < 1 || n_in > BD_MAX_SUB || n_out < 1 || n_out > BD_MAX_SUB || !bd_dual_ok(k, g)) return CAFEQ_ERR_INVALID_ARG;
  BdMaps mi, mo;
  BdMulti pi, po;
  memset(&pi, 0, sizeof(pi));
  memset(&po, 0, sizeof(po));
  for (int s = 0; s < n_in; ++s) {
    if (!make_map_bf16(&mi.x[s], in[s].X, in[s].p.d_in, in[s].p.d_out, in[s].ld, 128)) return CAFEQ_ERR_UNSUPPORTED;
    if (!make_map_bf16(&mi.t[s], in[s].Tb, k, (long long)in[s].nbT * k, k, bd_operator_rows(k, in[s].p))) return CAFEQ_ERR_UNSUPPORTED;
    pi.p[s] = in[s].p;
  }
  for (int s = n_in; s < BD_MAX_SUB; ++s) { mi.x[s] = mi.x[0]; mi.t[s] = mi.t[0]; }
  for (int s = 0; s < n_out; ++s) {
    if (!make_map_bf16(&mo.x[s], out[s].X, out[s].p.d_in, out[s].p.d_out, out[s].ld, 128)) return CAFEQ_ERR_UNSUPPORTED;
    if (!make_map_bf16(&mo.t[s], out[s].Tb, k, (long long)out[s].nbT * k, k, bd_operator_rows(k, out[s].p))) return CAFEQ_ERR_UNSUPPORTED;
    po.p[s] = out[s].p;
  }
  for (int s = n_out; s < BD_MAX_SUB; ++s) { mo.x[s] = mo.x[0]; mo.t[s] = mo.t[0]; }
  pi.n = n_in;
  po.n = n_out;
#define BD_DUAL(KK, GG) \
  if (k == KK && g == GG) return bd_launch_dual_t<KK, GG>(st, mi, pi, mo, po, overlap);
  BD_DUAL(128, 64)
  BD_DUAL(128, 128)
  BD_DUAL(256, 64)
  BD_DUAL(256, 128)
#undef BD_DUAL
  return CAFEQ_ERR_UNSUPPORTED;
}

// fp32 operator blocks -> bf16 in applied orientation (transposed when the role asks for T^T); k % 32 == 0, one 32 x 32 tile
// per CTA (grid: (blocks, k / 32, k / 32): only the first dimension holds any number of blocks), rows read and written along
// their elements.  Latency-bound: one load, one store
// (14 blocks of 256: 5 - 7 us with a strided walk and 64-bit divisions per element, 3 us here).
// paired (k = 32): blocks 2 i and 2 i + 1 become one 64 x 64 block, zeros off the diagonal.
__global__ void __launch_bounds__(256) operator_to_bf16_kernel(const float* T, uint16_t* __restrict__ out, int k, int transpose,
                                                               int paired, const int32_t* status) {
  pdl_enter();
  if (cta_stopped(status)) return;
  __shared__ float tile[32][33];
  const size_t base = (size_t)blockIdx.x * k * k;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.z * 32;  // tile of the output
  const int i = threadIdx.x >> 3, j = (threadIdx.x & 7) * 4;
  const float* src = T + base + (transpose ? (size_t)(c0 + i) * k + r0 + j : (size_t)(r0 + i) * k + c0 + j);
  float v[4];
  if (((uintptr_t)T & 15) == 0) {
    const float4 q = ld_plain(reinterpret_cast<const float4*>(src));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = ld_plain(src + e);
  }
  if (transpose) {
#pragma unroll
    for (int e = 0; e < 4; ++e) tile[i][j + e] = v[e];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = tile[j + e][i];
  }
  uint32_t w[2];
#pragma unroll
  for (int e = 0; e < 2; ++e)
    w[e] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[2 * e])) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[2 * e + 1])) << 16);
  if (paired) {
    const int odd = blockIdx.x & 1;
    uint16_t* o = out + (size_t)(blockIdx.x >> 1) * 4096 + (odd * 32 + i) * 64 + j;
    *reinterpret_cast<uint2*>(o + odd * 32) = make_uint2(w[0], w[1]);
    *reinterpret_cast<uint2*>(o + (1 - odd) * 32) = make_uint2(0u, 0u);
    return;
  }
  *reinterpret_cast<uint2*>(out + base + (size_t)(r0 + i) * k + c0 + j) = make_uint2(w[0], w[1]);
}

// ------------------------------------------------------------------------------------------------
// Y = P o X on the input axis for few rows (decoding): bf16 operands, fp32 accumulation, the operator read once in fp32 and
// rounded on the way, so there is no conversion launch and no scratch.  Bound by latency: a CTA owns 32 output columns of one
// block and eight rows, so that 14 blocks of 256 are 112 CTAs (in the tensor-core pass they are 14, each loading its
// 128 KB operator through one TMA ring).  The operator tile and the rows go to shared memory as [contraction][column] and
// [contraction][row]; warp w takes an eighth of the contraction, its partial sums meet in shared memory.
// ------------------------------------------------------------------------------------------------
constexpr int AS_ROWS = 8, AS_MAX_ROWS = 64;
__global__ void __launch_bounds__(256) apply_small_kernel(const uint16_t* X, long long ld, const float* T,
                                                          uint16_t* __restrict__ Y, int rows, int d_in, int k, int r, int transposed,
                                                          const int32_t* status) {
  pdl_enter();
  if (cta_stopped(status)) return;
  __shared__ float ps[256 * 33];
  __shared__ float4 xs4[256 * AS_ROWS / 4];
  float* xs = reinterpret_cast<float*>(xs4);
  const int strips = k / 32;
  const int b = blockIdx.x / strips, n0 = (blockIdx.x - b * strips) * 32;
  const int t0 = blockIdx.y * AS_ROWS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* Tb = T + (size_t)(b / r) * k * k;
  if (transposed) {  // P[n][m] = T[m][n]: 8 threads per contraction row
#pragma unroll 8
    for (int m = tid >> 3; m < k; m += 32) {
      const int n = (tid & 7) * 4;
      const float4 q = ld_plain(reinterpret_cast<const float4*>(Tb + (size_t)m * k + n0 + n));
      float* d = ps + m * 33 + n;
      d[0] = round_to_bf16(q.x); d[1] = round_to_bf16(q.y); d[2] = round_to_bf16(q.z); d[3] = round_to_bf16(q.w);
    }
  } else {  // P[n][m] = T[n][m]: k / 4 threads per output column
    const int q4 = k / 4;
#pragma unroll 8
    for (int e = tid; e < 32 * q4; e += 256) {
      const int n = e / q4, m = (e - n * q4) * 4;
      const float4 q = ld_plain(reinterpret_cast<const float4*>(Tb + (size_t)(n0 + n) * k + m));
      float* d = ps + m * 33 + n;
      d[0] = round_to_bf16(q.x); d[33] = round_to_bf16(q.y); d[66] = round_to_bf16(q.z); d[99] = round_to_bf16(q.w);
    }
  }
  for (int m = tid; m < k; m += 256)
#pragma unroll
    for (int t = 0; t < AS_ROWS; ++t)
      xs[m * AS_ROWS + t] = (t0 + t < rows) ? bf16_bits_to_float(X[(long long)(t0 + t) * ld + (long long)b * k + m]) : 0.f;
  __syncthreads();
  float acc[AS_ROWS];
#pragma unroll
  for (int t = 0; t < AS_ROWS; ++t) acc[t] = 0.f;
  const int len = k / 8;
#pragma unroll 4
  for (int m = warp * len; m < (warp + 1) * len; ++m) {
    const float w = ps[m * 33 + lane];
    const float4 x0 = xs4[m * 2], x1 = xs4[m * 2 + 1];
    acc[0] = fmaf(w, x0.x, acc[0]); acc[1] = fmaf(w, x0.y, acc[1]); acc[2] = fmaf(w, x0.z, acc[2]); acc[3] = fmaf(w, x0.w, acc[3]);
    acc[4] = fmaf(w, x1.x, acc[4]); acc[5] = fmaf(w, x1.y, acc[5]); acc[6] = fmaf(w, x1.z, acc[6]); acc[7] = fmaf(w, x1.w, acc[7]);
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < AS_ROWS; ++t) ps[(warp * AS_ROWS + t) * 32 + lane] = acc[t];
  __syncthreads();
  float y = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) y += ps[(w * AS_ROWS + warp) * 32 + lane];
  if (t0 + warp < rows)
    Y[(long long)(t0 + warp) * d_in + (long long)b * k + n0 + lane] = __bfloat16_as_ushort(__float2bfloat16_rn(y));
}

}  // namespace cafeq
