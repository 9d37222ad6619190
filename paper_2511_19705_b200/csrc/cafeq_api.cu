// C-ABI entry points of the CafeQ optimisation path (declared in include/cafeq.h).
// Host side only validates arguments, carves the caller's workspace and enqueues kernels.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <type_traits>
#include <vector>

#include "cafeq.h"
#include "kernels_generic.cuh"
#include "kernels_fused.cuh"
#include "kernels_bwd.cuh"
#include "kernels_gemm.cuh"
#include "kernels_gemm2.cuh"
#include "kernels_small.cuh"
#include "kernels_kk.cuh"
#include "kernels_dense.cuh"
#include "kernels_rtn.cuh"

namespace cafeq {

// Process-wide count of kernel launches made by this library (read by benchmarks through
// cafeq_debug_launch_count; it has no effect on any result).
static std::atomic<long long> g_launches{0};
#define CQ_LAUNCH_IF(overlap, kernel, grid, block, smem, st, ...)       \
  do {                                                                  \
    g_launches.fetch_add(1, std::memory_order_relaxed);                 \
    launch_pdl_if(overlap, kernel, grid, block, smem, st, __VA_ARGS__); \
  } while (0)
#define CQ_LAUNCH(kernel, grid, block, smem, st, ...) CQ_LAUNCH_IF(true, kernel, grid, block, smem, st, __VA_ARGS__)

// Optional per-launch timing of selected kernels with CUDA events on the launching stream (benchmarks
// only; off unless cafeq_debug_timer_begin was called).  Kinds: 1 transform pass (shape-agnostic kernels),
// 2 sparse backward, 3 block inverse, 4 dense pair product, 5 fused tensor-core transform pass.
struct KernelTimer {
  std::vector<cudaEvent_t> a, b;
  std::vector<int> kind;
  int used = 0;
  bool on = false;
};
static KernelTimer g_kt;
static inline int kt_begin(int kind, cudaStream_t st) {
  if (!g_kt.on || g_kt.used >= (int)g_kt.a.size()) return -1;
  int i = g_kt.used++;
  g_kt.kind[i] = kind;
  cudaEventRecord(g_kt.a[i], st);
  return i;
}
static inline void kt_end(int i, cudaStream_t st) {
  if (i >= 0) cudaEventRecord(g_kt.b[i], st);
}

// ------------------------------------------------------------------------------------------------
// workspace carving
// ------------------------------------------------------------------------------------------------
struct Bump {
  char* base;
  size_t cap, used;
  bool overflow;
  Bump(void* b, size_t c) : base((char*)b), cap(c), used(0), overflow(false) {}
  // (base == nullptr: nothing is handed out, `used` still adds up -- the size queries run the same carving code)
  template <typename T>
  T* take(size_t count) {
    size_t bytes = (count * sizeof(T) + 255) & ~(size_t)255;
    if (!base || used + bytes > cap) { overflow = true; used += bytes; return nullptr; }
    T* p = (T*)(base + used);
    used += bytes;
    return p;
  }
};

static inline int grid_for(long long n, int threads = 256, int cap = 148 * 16) {
  long long b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (int)b;
}

static inline float qmax_of(int bits) { return (float)((1 << (bits - 1)) - 1); }

struct Geo {  // derived geometry of one descriptor
  int d_out, d_in, g, ng, k, r, axis, nbq, nbT;
  long long ld, n;
};

static int make_geo(const cafeq_matrix_desc* d, Geo* o, bool need_transform) {
  if (!d || d->struct_size != sizeof(cafeq_matrix_desc)) return CAFEQ_ERR_INVALID_ARG;
  if (d->d_out <= 0 || d->d_in <= 0 || d->ld < d->d_in) return CAFEQ_ERR_INVALID_ARG;
  if (d->bits < 2 || d->bits > 8) return CAFEQ_ERR_INVALID_ARG;
  if (d->group < 0 || d->tblock < 0 || d->replicas < 1) return CAFEQ_ERR_INVALID_ARG;
  if (d->taxis != CAFEQ_AXIS_IN && d->taxis != CAFEQ_AXIS_OUT) return CAFEQ_ERR_INVALID_ARG;
  if (d->compute_prec != CAFEQ_PREC_BF16) return CAFEQ_ERR_UNSUPPORTED;
  o->d_out = d->d_out;
  o->d_in = d->d_in;
  o->ld = d->ld;
  o->n = (long long)d->d_out * d->d_in;
  o->g = d->group ? d->group : d->d_in;
  if (d->d_in % o->g) return CAFEQ_ERR_INVALID_ARG;
  o->ng = d->d_in / o->g;
  o->k = d->tblock;
  o->r = d->replicas;
  o->axis = d->taxis;
  o->nbq = 0;
  o->nbT = 0;
  if (o->k > 0) {
    int dim = (o->axis == CAFEQ_AXIS_IN) ? d->d_in : d->d_out;
    if (dim % o->k) return CAFEQ_ERR_INVALID_ARG;
    o->nbq = dim / o->k;
    if (o->nbq % o->r) return CAFEQ_ERR_INVALID_ARG;
    o->nbT = o->nbq / o->r;
    if (o->k > 1024) return CAFEQ_ERR_UNSUPPORTED;
  } else if (need_transform) {
    return CAFEQ_ERR_INVALID_ARG;
  }
  return CAFEQ_OK;
}

// ------------------------------------------------------------------------------------------------
// launch helpers
// ------------------------------------------------------------------------------------------------
static void launch_gemm(cudaStream_t st, const GemmArgs& g) {
  dim3 grid((g.N + 63) / 64, (g.M + 63) / 64, g.batch);
  if (g.a_bf16 && g.b_bf16) CQ_LAUNCH((gemm_kernel<true, true>), grid, 256, 0, st, g);
  else if (g.a_bf16) CQ_LAUNCH((gemm_kernel<true, false>), grid, 256, 0, st, g);
  else if (g.b_bf16) CQ_LAUNCH((gemm_kernel<false, true>), grid, 256, 0, st, g);
  else CQ_LAUNCH((gemm_kernel<false, false>), grid, 256, 0, st, g);
}

static GemmArgs gemm_defaults(const int32_t* status) {
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.divA = g.divB = g.divC = 1;
  g.alpha = 1.f;
  g.mode = GEMM_STORE;
  g.batch = 1;
  g.status = status;
  return g;
}

// Out = T o X along `axis`; X is bf16 (x_bf16) or fp32; T fp32 blocks [nbT,k,k]; transposed uses T^T.
static void launch_apply(cudaStream_t st, const void* X, int x_bf16, long long ldx, const Geo& G, const float* T,
                         int transposed, float* Out, long long ldo, int mode, double* sq, const int32_t* status,
                         float alpha = 1.f) {
  GemmArgs g = gemm_defaults(status);
  const int k = G.k;
  g.alpha = alpha;
  g.C = Out;
  g.mode = mode;
  g.sq = sq;
  g.batch = G.nbq;
  if (G.axis == CAFEQ_AXIS_IN) {
    g.M = G.d_out; g.N = k; g.K = k;
    g.A = X; g.a_bf16 = x_bf16; g.sAm = ldx; g.sAk = 1; g.sAb = k;
    g.B = T; g.b_bf16 = 0; g.sBb = (long long)k * k; g.divB = G.r;
    if (!transposed) { g.sBk = 1; g.sBn = k; } else { g.sBk = k; g.sBn = 1; }
    g.sCm = ldo; g.sCn = 1; g.sCb = k;
  } else {
    g.M = k; g.N = G.d_in; g.K = k;
    g.A = T; g.a_bf16 = 0; g.sAb = (long long)k * k; g.divA = G.r;
    if (!transposed) { g.sAm = k; g.sAk = 1; } else { g.sAm = 1; g.sAk = k; }
    g.B = X; g.b_bf16 = x_bf16; g.sBk = ldx; g.sBn = 1; g.sBb = (long long)k * ldx;
    g.sCm = ldo; g.sCn = 1; g.sCb = (long long)k * ldo;
  }
  int ti = kt_begin(1, st);
  launch_gemm(st, g);
  kt_end(ti, st);
}

// gT[b / r][i][j] += alpha * sum_free Gm[.., i] X[.., j]  (atomic accumulation; caller zeroes gT)
static void launch_opgrad(cudaStream_t st, const float* Gm, long long ldg, const void* X, int x_bf16, long long ldx,
                          const Geo& G, float* gT, int transpose_out, float alpha, const int32_t* status) {
  GemmArgs g = gemm_defaults(status);
  const int k = G.k;
  g.M = k; g.N = k; g.batch = G.nbq;
  g.A = Gm; g.a_bf16 = 0;
  g.B = X; g.b_bf16 = x_bf16;
  g.C = gT; g.sCb = (long long)k * k; g.divC = G.r;
  if (!transpose_out) { g.sCm = k; g.sCn = 1; } else { g.sCm = 1; g.sCn = k; }
  g.alpha = alpha;
  g.mode = GEMM_STORE | GEMM_ATOMIC;
  if (G.axis == CAFEQ_AXIS_IN) {
    g.K = G.d_out;
    g.sAm = 1; g.sAk = ldg; g.sAb = k;
    g.sBk = ldx; g.sBn = 1; g.sBb = k;
  } else {
    g.K = G.d_in;
    g.sAm = ldg; g.sAk = 1; g.sAb = (long long)k * ldg;
    g.sBk = 1; g.sBn = ldx; g.sBb = (long long)k * ldx;
  }
  launch_gemm(st, g);
}

// C[b] (op)= alpha * opA(A[b]) * opB(B[b]) for k x k blocks
static void launch_kk(cudaStream_t st, const float* A, int tA, const float* B, int tB, float* C, int nb, int k, float alpha,
                      int mode, const int32_t* status) {
  GemmArgs g = gemm_defaults(status);
  g.M = g.N = g.K = k;
  g.batch = nb;
  g.A = A; g.B = B; g.C = C;
  g.sAb = g.sBb = g.sCb = (long long)k * k;
  if (!tA) { g.sAm = k; g.sAk = 1; } else { g.sAm = 1; g.sAk = k; }
  if (!tB) { g.sBk = k; g.sBn = 1; } else { g.sBk = 1; g.sBn = k; }
  g.sCm = k; g.sCn = 1;
  g.alpha = alpha;
  g.mode = mode;
  launch_gemm(st, g);
}

static void launch_inverse(cudaStream_t st, const float* Mc, float* Minv, float* cnorm, int nb, int k, int32_t* status,
                           uint16_t* hi = nullptr, uint16_t* lo = nullptr, uint16_t* thi = nullptr, uint16_t* tlo = nullptr) {
  int ti = kt_begin(3, st);
  if (k == 32) CQ_LAUNCH(small_inverse_kernel<32>, nb, 256, 0, st, Mc, Minv, cnorm, hi, lo, thi, tlo, status);
  else if (k == 64) CQ_LAUNCH(small_inverse_kernel<64>, nb, 256, 0, st, Mc, Minv, cnorm, hi, lo, thi, tlo, status);
  else {  // (no splits)
    const int threads = k * k >= 1024 ? 1024 : ((k * k + 31) / 32) * 32;
    CQ_LAUNCH(block_inverse_kernel, nb, threads, (size_t)3 * k * sizeof(float), st, Mc, Minv, cnorm, k, status);
  }
  kt_end(ti, st);
}

// ------------------------------------------------------------------------------------------------
// k x k algebra on the tensor cores: split-precision products and the Newton-Schulz inverse
// ------------------------------------------------------------------------------------------------
struct KkWS {  // bf16 scratch, each [nbT * k * k]
  uint16_t *Ab;              // bf16(M)
  uint16_t *Xh, *Xl;         // splits of the inverse, and transposed:
  uint16_t *XTh, *XTl;       // (blocks of 32 and 64 only)
  uint16_t *RTh, *RTl, *Ph, *Pl, *Qh, *Ql;
  int* redo_total;           // optional running count of blocks recomputed by elimination (never cleared by a step)
  bool mn;                   // the inverse was refined on row-major arrays only (blocks of 128 and 256): XTh / XTl are not maintained
};
// Fused kernel (ns_block_kernel): rounds at most, and the squared residual before an update that makes it the last one.
// Warm: below 1e-2 before, hence below 1e-4 after it (the acceptance test of the elimination fall-back).  Cold starts are
// paid once per run: they go on to 1e-3 (1e-6 after the update, and up to 4e-6 from the update's single term).
constexpr int NS_WARM_ROUNDS = 6, NS_COLD_ROUNDS = 10;
constexpr double NS_GATE2 = 1e-4, NS_COLD_GATE2 = 1e-6;

static void launch_operator_bf16(cudaStream_t st, const float* T, uint16_t* out, int k, int nb, int transpose, int32_t* status,
                                 int paired = 0) {
  CQ_LAUNCH(operator_to_bf16_kernel, dim3(nb, k / 32, k / 32), 256, 0, st, T, out, k, transpose, paired, status);
}

static bool kk_fast(int k) { return k == 64 || k == 128 || k == 256; }

// layer: what the layer step uses of it
static void carve_kk(Bump& b, int nbT, int k, KkWS* w, bool layer = false) {
  const size_t kk = (size_t)nbT * k * k;
  memset(w, 0, sizeof(*w));
  for (uint16_t** p : {&w->Ab, &w->Xh, &w->Xl, &w->Pl}) *p = b.take<uint16_t>(kk);
  if (layer) return;
  for (uint16_t** p : {&w->XTh, &w->XTl, &w->RTh, &w->RTl, &w->Ph, &w->Qh, &w->Ql}) *p = b.take<uint16_t>(kk);
}

// C[b] = alpha * sum_t A_t[b] B_t[b]^T + beta * C0[b] + gamma * I for nb blocks of k x k; operands bf16 [nb*k, k]
static int launch_kk_tc(cudaStream_t st, int nterms, const uint16_t* const* A, const uint16_t* const* B, int nb, int k,
                        float alpha, float beta, float gamma, const float* C0, float* C, uint16_t* Chi, uint16_t* Clo,
                        uint16_t* Cthi, uint16_t* Ctlo, double* sq, int32_t* status, int sq_stride = 1, int a_mn = 0, int b_mn = 0) {
  TgOperand oa[TG_MAX_TERMS], ob[TG_MAX_TERMS];
  for (int t = 0; t < nterms; ++t) {
    oa[t] = TgOperand{A[t], (long long)nb * k, k, k};
    ob[t] = TgOperand{B[t], (long long)nb * k, k, k};
  }
  TgParams p;
  memset(&p, 0, sizeof(p));
  p.M = p.N = p.K = k;
  p.batch = nb;
  p.nterms = nterms;
  p.rowsA_per_batch = p.rowsB_per_batch = k;
  p.divA = 1;
  p.alpha = alpha; p.beta = beta; p.gamma = gamma;
  p.C0 = C0; p.ldc0 = k; p.sC0b = (long long)k * k;
  p.C = C; p.ldc = k; p.sCb = (long long)k * k;
  p.Chi = Chi; p.Clo = Clo; p.Cthi = Cthi; p.Ctlo = Ctlo;
  p.sq = sq; p.sq_stride = sq_stride;
  p.status = status;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (tb_supported(k, nterms)) {
    const int rc = tb_launch(st, nterms, A, B, a_mn, b_mn, (long long)nb * k, (long long)nb * k, k, p);
    if (rc != CAFEQ_ERR_UNSUPPORTED) return rc;
  }
  if (a_mn || b_mn) return CAFEQ_ERR_UNSUPPORTED;  // the tiled kernel takes K-major operands only
  return tg_launch(st, oa, ob, p);
}

static void launch_split(cudaStream_t st, const float* X, int k, long long n, uint16_t* hi, uint16_t* lo, uint16_t* thi,
                         uint16_t* tlo, const int32_t* status) {
  dim3 grid(k / 32, k / 32, (unsigned)(n / ((long long)k * k)));
  CQ_LAUNCH(split_bf16_kernel, grid, dim3(32, 8), 0, st, X, k, hi, lo, thi, tlo, status);
}

// Batched products of 256 x 256 with their contraction in parts (tg_launch_split; parts: scratch for K / 256 * reps * batch of them), summed
// into out and, optionally, its splits.
// Against tiles with the whole contraction each (8 CTAs a block, K / 64 chunks in a row, some 0.8 us a chunk) the parts cost a longer
// first tile, a launch, and a trip of 256 KB each.  Measured, tiles -> parts, Eq. 3 straight-through: blocks x K 1 x 256 188.7 -> 193.0
// us, 4 x 700 205 -> 205, 4 x 1024 214 -> 209, 14 x 1024 225 -> 230, 8 x 1500 221 -> 212, 74 x 512 301 -> 304, 14 x 4096 348 -> 312;
// Eq. 5: 16 x 1024 359 -> 364, 8 x 2048 327 -> 313, 8 x 3584 with two replicas 792 -> 729.
static bool split_wanted(int k, int K, int batch, int reps) {
  return k == 256 && K >= 256 && K / 64 >= 12 + batch * reps * t2_slices(batch * reps, K) / 8;
}
static int launch_split_product(cudaStream_t st, int na, const TgOperand* A, int nb, const TgOperand* B, int K, int batch, int reps, int mn,
                                float* parts, float* out, uint16_t* hi, uint16_t* lo, int32_t* status) {
  int n = 0;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  const int rc = tg_launch_split(st, na, A, nb, B, K, batch, reps, mn, 1.f, parts, &n, status);
  if (rc) return rc;
  CQ_LAUNCH(sum_parts_kernel, 64u * (unsigned)batch, 256, 0, st, parts, n, out, hi, lo, status);
  return CAFEQ_OK;
}

// Minv = inv(bf16(M)).  k = 128, 256: Newton-Schulz iteration X <- X + X (I - A X) on the tensor cores, every round of a block
// in one launch, from X0 = A^T (cold: right for the near-orthogonal transforms the method starts from) or from the caller's
// previous inverse (warm); a warm start runs as many rounds as the step size calls for (a block whose residual ||I - A X||_F
// was below 1e-2 before an update, 1e-4 after it, stops); a residual that does not become small falls back to elimination.
// k = 32, 64: elimination, which takes less than one round's launches there.  Leaves fp32 Minv in X and its bf16 splits in
// w.Xh / Xl (and XTh / XTl unless w.mn).
// eq4 (k = 128, 256): where the kernel puts the column norms / group weights, and what it ticks.
static int ns_inverse(cudaStream_t st, const float* Mc, float* X, int nb, int k, bool warm, KkWS& w, int32_t* status,
                      bool prepped = false, bool splits_kept = false, const NsParams* eq4 = nullptr, bool overlap = true) {
  w.mn = tb_supported(k, 2);
  if (!w.mn) {
    launch_inverse(st, Mc, X, nullptr, nb, k, status, w.Xh, w.Xl, w.XTh, w.XTl);
    return CAFEQ_OK;
  }
  int ti = kt_begin(3, st);
  if (!prepped) launch_operator_bf16(st, Mc, w.Ab, k, nb, 0, status);  // (otherwise the step's set-up has written it)
  // (splits_kept: the splits of X that the previous call left are still there)
  if (!warm) CQ_LAUNCH(ns_cold_start_kernel, dim3(k / 32, k / 32, nb), dim3(32, 8), 0, st, w.Ab, k, w.Xh, w.Xl, status);
  else if (!splits_kept) launch_split(st, X, k, (long long)nb * k * k, w.Xh, w.Xl, nullptr, nullptr, status);
  NsParams np;
  memset(&np, 0, sizeof(np));
  if (eq4) np = *eq4;
  np.max_rounds = warm ? NS_WARM_ROUNDS : NS_COLD_ROUNDS;
  np.gate2 = warm ? NS_GATE2 : NS_COLD_GATE2;
  np.accept2 = NS_GATE2;
  np.redo_count = w.redo_total;
  np.status = status;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  const int rc = ns_block_launch(st, w.Ab, w.Xh, w.Xl, X, nb, k, np, overlap);
  kt_end(ti, st);
  return rc;
}

// G -= X^T Gx X^T for every block; X = Minv.  k = 128, 256: on the tensor cores from its splits in w, three-term
// products; 32, 64: in fp32.  Gx = dL/dMinv: fp32 [nb, k, k], or (scaled) formed from X by the kernel itself.
static int minv_path_tc(cudaStream_t st, const float* X, const float* Gx, float* G, int nb, int k, KkWS& w, int32_t* status,
                        const ChainParams* scaled = nullptr, bool overlap = true) {
  ChainParams cp;
  memset(&cp, 0, sizeof(cp));
  if (scaled) cp = *scaled;
  if (w.mn) {
    cp.G = Gx;
    cp.status = status;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return kk_chain_launch(st, KK_MINV_PATH, w.Xh, w.Xl, G, nb, k, cp, overlap);
  }
  if (k == 32) CQ_LAUNCH(small_chain_kernel<32>, nb, 64, 0, st, X, Gx, cp.A[0], cp.Agrp[0], cp.g[0], cp.scale[0], G, status);
  else CQ_LAUNCH(small_chain_kernel<64>, nb, 256, 0, st, X, Gx, cp.A[0], cp.Agrp[0], cp.g[0], cp.scale[0], G, status);
  return CAFEQ_OK;
}

// Orthonormality penalty of nb blocks from the splits of the fp32 parameters (fused kernel, k = 128 / 256):
// sq[b * sq_stride] += ||M_b M_b^T - I||_F^2 and, with want_out, out = (M M^T - I) M.
static int penalty_tc(cudaStream_t st, const uint16_t* Mh, const uint16_t* Ml, float* out, bool want_out, double* sq, int sq_stride,
                      int nb, int k, int32_t* status, bool overlap = true) {
  ChainParams cp;
  memset(&cp, 0, sizeof(cp));
  cp.sq = sq; cp.sq_stride = sq_stride;
  cp.want_out = want_out ? 1 : 0;
  cp.status = status;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return kk_chain_launch(st, KK_PENALTY, Mh, Ml, out, nb, k, cp, overlap);
}

static void launch_absmax(cudaStream_t st, const float* U, long long ld, const Geo& G, float* a, float* usel, int* idx,
                          int32_t* status) {
  long long warps = (long long)G.d_out * G.ng;
  long long blocks = (warps * 32 + 255) / 256;
  CQ_LAUNCH(absmax_kernel, (unsigned)blocks, 256, 0, st, U, ld, G.d_out, G.ng, G.g, a, usel, idx, status);
}

// Group quantiser of an fp32 matrix U [rows, ng g] (pitch ld; Delta / Uhat share it): maxima, signed arg-max values, arg-max
// positions, scales, residual, dequantised values, codes -- each optional except a / usel / idx.
template <typename SRC>
static bool launch_group_quant_vec(cudaStream_t st, const SRC* U, long long ld, int rows, int ng, int g, float qmax, const void* offsets,
                                   int off_kind, float* a, float* usel, int* idx, float* Delta, float* Uhat, int8_t* codes, float* scales,
                                   int32_t* status) {
  const long long groups = (long long)rows * ng;
  if (g % 4 || g > 16384 || ld % 4 || ((uintptr_t)U & (4 * sizeof(SRC) - 1)) || (((uintptr_t)Delta | (uintptr_t)Uhat) & 15) ||
      ((uintptr_t)codes & 3))
    return false;
#define GQ(L, N)                                                                                                              \
  CQ_LAUNCH((group_quant_kernel<L, N, SRC>), (unsigned)((groups * L + 255) / 256), 256, 0, st, U, ld, rows, ng, g, qmax, offsets, off_kind, \
            a, usel, idx, Delta, Uhat, codes, scales, status)
  // Four vectors of four a lane where the group has them (two in groups of 32): a lane's loads are in flight together, and the
  // reduction over lanes, fifteen shuffles for four values at one vector a lane of 32, is nine for sixteen.  Where that leaves less than
  // 512 threads an SM (2^20 entries) a lane has one (Eq. 5's straight-through gradient of 512 x 1024 with blocks of 64: four vectors 166.5
  // us a call, one 164.5; Eq. 3's of 1024 x 1024 192.5 and 194.5).  Above eight vectors a lane, the whole CTA.
  const bool few = groups * g < 1ll << 20;
  if (few && g <= 32) GQ(8, 1);
  else if (few && g <= 64) GQ(16, 1);
  else if (few && g <= 128) GQ(32, 1);
  else if (few && g <= 256) GQ(32, 2);
  else if (g <= 32) GQ(4, 2);
  else if (g <= 64) GQ(4, 4);
  else if (g <= 128) GQ(8, 4);
  else if (g <= 256) GQ(16, 4);
  else if (g <= 512) GQ(32, 4);
  else if (g <= 1024) GQ(32, 8);
  else if (g <= 2048) GQ(256, 2);
  else if (g <= 4096) GQ(256, 4);
  else if (g <= 8192) GQ(256, 8);
  else GQ(256, 16);
#undef GQ
  return true;
}
static void launch_group_quant(cudaStream_t st, const float* U, long long ld, int rows, int ng, int g, float qmax, const void* offsets,
                               int off_kind, float* a, float* usel, int* idx, float* Delta, float* Uhat, int8_t* codes, float* scales,
                               int32_t* status) {
  const long long groups = (long long)rows * ng;
  if (launch_group_quant_vec<float>(st, U, ld, rows, ng, g, qmax, offsets, off_kind, a, usel, idx, Delta, Uhat, codes, scales, status)) return;
  CQ_LAUNCH(absmax_kernel, (unsigned)((groups * 32 + 255) / 256), 256, 0, st, U, ld, rows, ng, g, a, usel, idx, status);
  if (Delta || Uhat || codes)
    CQ_LAUNCH(quant_kernel, grid_for((long long)rows * ng * g), 256, 0, st, U, ld, rows, ng * g, g, a, qmax, offsets, off_kind, Delta, Uhat,
              codes, status);
  if (scales) CQ_LAUNCH(scales_kernel, grid_for(groups), 256, 0, st, a, scales, groups, qmax, status);
}

// gm: the (row, group) records are group-major (written by the fused pass) instead of row-major
static void launch_scatter(cudaStream_t st, const void* W, const Geo& G, const float* coef, const int* idx, float* gT,
                           int transpose_out, const int32_t* status, int gm) {
  const int k = G.k;
  int ti = kt_begin(2, st);
  // block sizes 128 / 256: a dense product on the tensor cores whose left operand holds the routed coefficients
  if (bw_supported(G.axis == CAFEQ_AXIS_IN, G.d_out, G.d_in, G.ld, k, G.g, W)) {
    BwParams bp;
    memset(&bp, 0, sizeof(bp));
    bp.d_out = G.d_out; bp.d_in = G.d_in; bp.g = G.g; bp.ng = G.ng; bp.r = G.r;
    bp.gm = gm; bp.transpose_out = transpose_out;
    bp.coef = coef; bp.idx = idx; bp.gradT = gT;
    bp.status = const_cast<int32_t*>(status);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (bw_launch(st, G.axis == CAFEQ_AXIS_IN, k, W, G.ld, bp) == CAFEQ_OK) {
      kt_end(ti, st);
      return;
    }
    g_launches.fetch_sub(1, std::memory_order_relaxed);
  }
  const bool aligned = ((uintptr_t)W % 4 == 0) && (G.ld % 2 == 0);
  const int nG = (k >= G.g) ? k / G.g : 1;  // groups of one row inside one block (g | k or k | g on this path)
  if (kk_fast(k) && G.axis == CAFEQ_AXIS_IN && (k % G.g == 0 || G.g % k == 0) && nG <= 8 && ((uintptr_t)W % 16 == 0) &&
      (G.ld % 8 == 0)) {
    // 8 strip columns per thread at least: strip 32 at k = 256 (one thread per target row), 64 otherwise
    const int strip = (k == 256) ? 32 : 64;
    const int strips = k / strip;
    int rows_per = SCB_MAXP / nG;
    if (rows_per > 2048) rows_per = 2048;
    // enough CTAs to fill the machine a few times over, but never more rows than the record buffer holds
    int want = (148 * 4 + G.nbq * strips - 1) / (G.nbq * strips);
    int rp2 = (G.d_out + want - 1) / want;
    rp2 = ((rp2 + 31) / 32) * 32;
    if (rp2 < rows_per) rows_per = rp2;
    if (rows_per < 32) rows_per = 32;
    const int splits = (G.d_out + rows_per - 1) / rows_per;
    dim3 grid(G.nbq, strips, splits);
    const size_t sh = (size_t)k * (strip + 1) * 4 + (size_t)SCB_MAXP * 6;
    {  // the attribute is per device: set it on every call (cheap)
      cudaFuncSetAttribute(scatter_in_bucket_kernel<256, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * 33 * 4 + SCB_MAXP * 6);
      cudaFuncSetAttribute(scatter_in_bucket_kernel<128, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 65 * 4 + SCB_MAXP * 6);
      cudaFuncSetAttribute(scatter_in_bucket_kernel<64, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 65 * 4 + SCB_MAXP * 6);
    }
#define SC_INB(KV, SV)                                                                                                   \
  CQ_LAUNCH((scatter_in_bucket_kernel<KV, SV>), grid, 256, sh, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, G.g, G.r, nG, coef, \
            idx, gT, transpose_out, rows_per, status, gm)
    if (k == 64) SC_INB(64, 64);
    else if (k == 128) SC_INB(128, 64);
    else SC_INB(256, 32);
#undef SC_INB
    kt_end(ti, st);
    return;
  }
  if (k % SC2_JS == 0 && k <= 256 && aligned && G.axis == CAFEQ_AXIS_IN && (k % G.g == 0 || G.g % k == 0) &&
      (nG == 1 || nG == 2 || nG == 4)) {
    {
      cudaFuncSetAttribute(scatter_in_strip_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * SC2_JS * 4);
      cudaFuncSetAttribute(scatter_in_strip_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * SC2_JS * 4);
      cudaFuncSetAttribute(scatter_in_strip_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * SC2_JS * 4);
    }
    const int strips = k / SC2_JS;
    int splits = (148 * 3 + G.nbq * strips - 1) / (G.nbq * strips);
    if (splits < 1) splits = 1;
    int rows_per = (G.d_out + splits - 1) / splits;
    rows_per = ((rows_per + 31) / 32) * 32;
    splits = (G.d_out + rows_per - 1) / rows_per;
    dim3 grid(G.nbq, strips, splits);
    const size_t sh = (size_t)k * SC2_JS * 4;
#define SC_IN(NGV)                                                                                                       \
  CQ_LAUNCH(scatter_in_strip_kernel<NGV>, grid, 256, sh, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, G.g, k, G.r, coef, idx, \
            gT, transpose_out, rows_per, status, gm)
    if (nG == 1) SC_IN(1);
    else if (nG == 2) SC_IN(2);
    else SC_IN(4);
#undef SC_IN
    kt_end(ti, st);
    return;
  }
  if (kk_fast(k) && G.g % 4 == 0 && G.g <= 128 && ((uintptr_t)W % 8 == 0) && (G.ld % 4 == 0) && G.axis == CAFEQ_AXIS_OUT) {
    const int strips = k / SC2_JS;
    int splits = (148 * 4 + G.nbq * strips - 1) / (G.nbq * strips);
    if (splits < 1) splits = 1;
    int per = (G.ng + splits - 1) / splits;
    splits = (G.ng + per - 1) / per;
    dim3 grid(G.nbq, strips, splits);
    const size_t sh = (size_t)2 * SC2_JS * (G.g + 4) * 2;
#define SC_OUT(KV)                                                                                                      \
  CQ_LAUNCH(scatter_out_strip_kernel<KV>, grid, 256, sh, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, G.g, G.r, coef, idx, gT, \
            transpose_out, per, status, gm)
    if (k == 64) SC_OUT(64);
    else if (k == 128) SC_OUT(128);
    else SC_OUT(256);
#undef SC_OUT
    kt_end(ti, st);
    return;
  }
  size_t sh = (size_t)k * SCATTER_JS * sizeof(float);
  if (sh > 48 * 1024) {
    cudaFuncSetAttribute(scatter_in_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    cudaFuncSetAttribute(scatter_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  }
  int strips = (k + SCATTER_JS - 1) / SCATTER_JS;
  if (G.axis == CAFEQ_AXIS_IN) {
    int want = (148 * 4) / (G.nbq * strips) + 1;
    int splits = want < 1 ? 1 : want;
    int rows_per = (G.d_out + splits - 1) / splits;
    if (rows_per < 8) rows_per = 8;
    splits = (G.d_out + rows_per - 1) / rows_per;
    dim3 grid(G.nbq, strips, splits);
    CQ_LAUNCH(scatter_in_kernel, grid, 256, sh, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, G.g, k, G.r, coef, idx, gT,
                                             transpose_out, rows_per, status, gm);
  } else {
    int want = (148 * 4) / (G.nbq * strips) + 1;
    int splits = want < 1 ? 1 : want;
    int per = (G.ng + splits - 1) / splits;
    if (per < 1) per = 1;
    splits = (G.ng + per - 1) / per;
    dim3 grid(G.nbq, strips, splits);
    CQ_LAUNCH(scatter_out_kernel, grid, 256, sh, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, G.g, k, G.r, coef, idx, gT,
                                              transpose_out, per, status, gm);
  }
  kt_end(ti, st);
}

__global__ void bf16_to_f32_kernel(const uint16_t* W, long long ld, int rows, int cols, float* __restrict__ U) {
  pdl_enter();
  const long long n = (long long)rows * cols;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    int row = (int)(e / cols), col = (int)(e - (long long)row * cols);
    U[e] = bf16_bits_to_float(W[row * ld + col]);
  }
}

__global__ void resid_sq_kernel(float* __restrict__ R, const float* P, long long n, double* acc,
                                const int32_t* status) {
  pdl_enter();
  if (cta_stopped(status)) return;
  __shared__ double red[32];
  double local = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    float v = R[i] - P[i];
    R[i] = v;
    local += (double)v * v;
  }
  double s = block_sum_double(local, red);
  if (threadIdx.x == 0) atomicAdd(acc, s);
}

// ------------------------------------------------------------------------------------------------
// per-matrix scratch
// ------------------------------------------------------------------------------------------------
struct MatWS {
  uint16_t *Tb, *Dbf;  // fused pass: bf16 operator blocks (applied orientation) and bf16 residual
  float *U, *D, *E;
  float *a, *usel, *coef, *cw, *agrp;
  int* idx;
};

// lean: the matrix goes through the fused tensor-core pass and nothing but the per-group records leaves it (Eq. 4 /
// LogSumExp steps without the quantised loss): no matrix-sized scratch at all.
static void carve_matrix(Bump& b, const Geo& G, MatWS* w, bool need_E, bool lean = false) {
  w->Tb = b.take<uint16_t>((size_t)(G.nbT > 0 ? G.nbT : 1) * (G.k > 0 ? G.k : 1) * (G.k > 0 ? G.k : 1));
  w->Dbf = lean ? nullptr : b.take<uint16_t>(G.n);
  w->U = lean ? nullptr : b.take<float>(G.n);
  w->D = lean ? nullptr : b.take<float>(G.n);
  w->E = (need_E && !lean) ? b.take<float>(G.n) : nullptr;
  size_t rows_ng = (size_t)G.d_out * G.ng;
  w->a = b.take<float>(rows_ng);
  w->usel = b.take<float>(rows_ng);
  w->idx = b.take<int>(rows_ng);
  w->coef = b.take<float>(rows_ng);
  w->cw = b.take<float>((size_t)(G.ng > G.d_out ? G.ng : G.d_out));
  w->agrp = b.take<float>((size_t)G.ng);
}

// One fused tensor-core pass (see kernels_fused.cuh); returns false when the shape is not covered.
static bool fused_pass(cudaStream_t st, const void* X, long long ldx, const Geo& G, const float* Top, int transposed,
                       uint16_t* Tb, BdParams p, int32_t* status, const uint16_t* Tb_ready = nullptr, void* pair_scratch = nullptr) {
  const int form = (G.axis == CAFEQ_AXIS_IN) ? BD_IN : BD_OUT;
  // blocks of 32 go through as pairs on the diagonal of blocks of 64, which take twice the room: 4 bytes per operator entry that
  // the pass leaves alone (pair_scratch; null: not in pairs)
  const int two = (form == BD_IN && G.k == 32 && G.r == 1 && pair_scratch) ? 1 : 0;
  const int k = two ? 64 : G.k, nbT = two ? G.nbT / 2 : G.nbT;
  if (!bd_supported(form, G.d_out, G.d_in, ldx, k, G.g, X)) return false;
  if (two) Tb = (uint16_t*)pair_scratch;
  if (Tb_ready && !transposed && !two) Tb = const_cast<uint16_t*>(Tb_ready);  // bf16 operator already in applied orientation
  else launch_operator_bf16(st, Top, Tb, G.k, G.nbT, transposed, status, two);
  p.d_out = G.d_out;
  p.d_in = G.d_in;
  p.r = G.r;
  p.pairs = two;
  p.status = status;
  int ti = kt_begin(5, st);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  int rc = bd_launch(st, form, k, G.g, X, ldx, Tb, nbT, p);
  kt_end(ti, st);
  return rc == CAFEQ_OK;
}

static bool tc_apply_ok(int k) { return k == 32 || kk_fast(k); }

// U = T o W in fp32 as one-term batched products on the tensor cores (bf16 x bf16 products are exact, fp32
// accumulation: the same arithmetic as the fused pass).  Tb: bf16 operator blocks in applied orientation
// [nbT k, k].
static bool apply_tc(cudaStream_t st, const void* W, const Geo& G, const uint16_t* Tb, float* U, int32_t* status) {
  const int k = G.k;
  if (!tc_apply_ok(k) || ((uintptr_t)W & 15) || (G.ld % 8) || (G.d_in % 4)) return false;
  TgOperand oa[1], ob[1];
  TgParams p;
  memset(&p, 0, sizeof(p));
  p.nterms = 1; p.K = k; p.batch = G.nbq; p.alpha = 1.f;
  p.divA = 1;
  p.C = U; p.ldc = G.d_in;
  p.status = status;
  if (G.axis == CAFEQ_AXIS_IN) {
    oa[0] = TgOperand{W, G.d_out, G.d_in, G.ld};
    ob[0] = TgOperand{Tb, (long long)G.nbT * k, k, k};
    p.M = G.d_out; p.N = k;
    p.rowsA_per_batch = 0; p.colsA_per_batch = k;
    p.rowsB_per_batch = k; p.divB = G.r;
    p.sCb = k;
  } else {  // the contraction runs down the rows of W as they are stored
    oa[0] = TgOperand{Tb, (long long)G.nbT * k, k, k};
    ob[0] = TgOperand{W, G.d_out, G.d_in, G.ld};
    p.M = k; p.N = G.d_in;
    p.b_mn = 1;
    p.rowsA_per_batch = k; p.divA = G.r;
    p.rowsB_per_batch = k;
    p.sCb = (long long)k * G.d_in;
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return tg_launch(st, oa, ob, p) == CAFEQ_OK;
}

// U = T o W, group absmax / arg-max, and (optionally) the quantiser outputs.  Returns true when the fused
// tensor-core pass ran (then the residual is in w.Dbf as bf16 instead of w.D as fp32, and U is not stored).
// T_rounded: scratch for the bf16 rounding of Tc where Tc is not rounded yet (the tensor-core paths round it themselves).
// pair_scratch: see fused_pass.
static bool forward_quant(cudaStream_t st, const void* W, const Geo& G, int bits, const float* Tc, int transposed,
                          const MatWS& w, const void* offsets, int off_kind, bool want_delta, float* Uhat, int8_t* codes,
                          float* scales, int32_t* status, bool allow_fused, const BdParams* surr = nullptr,
                          const uint16_t* Tb_ready = nullptr, float* T_rounded = nullptr, void* pair_scratch = nullptr) {
  if (Tc && allow_fused && off_kind == CAFEQ_OFFSETS_NONE && !Uhat) {
    BdParams p;
    memset(&p, 0, sizeof(p));
    if (surr) p = *surr;
    p.epi = EPI_ABSMAX | (want_delta ? EPI_DELTA : 0) | (codes ? EPI_CODES : 0) | (surr ? EPI_SURR : 0);
    p.qmax = qmax_of(bits);
    p.a = w.a; p.usel = w.usel; p.idx = w.idx;
    p.delta = w.Dbf; p.codes = codes; p.scales = scales;
    if (fused_pass(st, W, G.ld, G, Tc, transposed, w.Tb, p, status, Tb_ready, pair_scratch)) return true;
  }
  if (!w.U) return false;  // lean workspace: there is no scratch for the shape-agnostic kernels (callers check first)
  bool applied = false;
  if (Tc && allow_fused) {  // (allow_fused is off when the caller asked for the shape-agnostic kernels)
    const uint16_t* Tb = (Tb_ready && !transposed) ? Tb_ready : w.Tb;
    if (Tb == w.Tb && tc_apply_ok(G.k)) launch_operator_bf16(st, Tc, w.Tb, G.k, G.nbT, transposed, status);
    applied = apply_tc(st, W, G, Tb, w.U, status);
  }
  if (applied) {
  } else if (Tc) {
    if (T_rounded) {
      const long long kk = (long long)G.nbT * G.k * G.k;
      CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, Tc, T_rounded, kk, nullptr);
    }
    launch_apply(st, W, 1, G.ld, G, T_rounded ? T_rounded : Tc, transposed, w.U, G.d_in, GEMM_STORE, nullptr, status);
  } else CQ_LAUNCH(bf16_to_f32_kernel, grid_for(G.n), 256, 0, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, w.U);
  launch_group_quant(st, w.U, G.d_in, G.d_out, G.ng, G.g, qmax_of(bits), offsets, off_kind, w.a, w.usel, w.idx, want_delta ? w.D : nullptr,
                     Uhat, codes, scales, status);
  return false;
}

}  // namespace cafeq

#include "pair_dense.cuh"

using namespace cafeq;

// ------------------------------------------------------------------------------------------------
extern "C" const char* cafeq_status_string(int s) {
  switch (s) {
    case CAFEQ_OK: return "ok";
    case CAFEQ_ERR_INVALID_ARG: return "invalid argument";
    case CAFEQ_ERR_UNSUPPORTED: return "unsupported shape or mode";
    case CAFEQ_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case CAFEQ_ERR_CUDA: return "CUDA launch failed";
    case CAFEQ_ERR_SINGULAR: return "singular transform block";
    case CAFEQ_ERR_NONFINITE: return "non-finite value";
    case CAFEQ_ERR_TIMEOUT: return "bounded device wait expired";
    case CAFEQ_ERR_TOO_LARGE: return "problem needs more scratch than the built-in buffer holds";
    default: return "unknown status";
  }
}

extern "C" int cafeq_version(void) { return 100; }

extern "C" long long cafeq_debug_launch_count(void) { return g_launches.load(); }

extern "C" int cafeq_set_overlap_mode(int overlapped) {
  if (overlapped != 0 && overlapped != 1) return CAFEQ_ERR_INVALID_ARG;
  g_tg_min_ctas.store(overlapped ? 28 : 96, std::memory_order_relaxed);
  g_bd_min_tiles.store(overlapped ? 14 : 1, std::memory_order_relaxed);
  g_bw_min_tiles.store(overlapped ? 14 : 6, std::memory_order_relaxed);
  return CAFEQ_OK;
}

extern "C" int cafeq_debug_wait_probe(unsigned long long limit_ns, int32_t* status, int* result, void* stream) {
  if (!status || !result) return CAFEQ_ERR_INVALID_ARG;
  CQ_LAUNCH(wait_probe_kernel, 1, 32, 0, (cudaStream_t)stream, (uint64_t)limit_ns, status, result);
  return cudaGetLastError() == cudaSuccess ? CAFEQ_OK : CAFEQ_ERR_CUDA;
}

extern "C" int cafeq_debug_timer_begin(int capacity) {
  if (capacity < 0 || g_kt.on) return CAFEQ_ERR_INVALID_ARG;
  g_kt.a.resize(capacity);
  g_kt.b.resize(capacity);
  g_kt.kind.assign(capacity, 0);
  for (int i = 0; i < capacity; ++i) {
    if (cudaEventCreate(&g_kt.a[i]) != cudaSuccess || cudaEventCreate(&g_kt.b[i]) != cudaSuccess) return CAFEQ_ERR_CUDA;
  }
  g_kt.used = 0;
  g_kt.on = true;
  return CAFEQ_OK;
}

extern "C" int cafeq_debug_timer_read(float* ms, int* kinds, int* count) {
  if (!g_kt.on || !ms || !kinds || !count) return CAFEQ_ERR_INVALID_ARG;
  int rc = CAFEQ_OK;
  for (int i = 0; i < g_kt.used; ++i) {
    if (cudaEventSynchronize(g_kt.b[i]) != cudaSuccess || cudaEventElapsedTime(&ms[i], g_kt.a[i], g_kt.b[i]) != cudaSuccess)
      rc = CAFEQ_ERR_CUDA;
    kinds[i] = g_kt.kind[i];
  }
  *count = g_kt.used;
  for (size_t i = 0; i < g_kt.a.size(); ++i) {
    cudaEventDestroy(g_kt.a[i]);
    cudaEventDestroy(g_kt.b[i]);
  }
  g_kt.a.clear();
  g_kt.b.clear();
  g_kt.kind.clear();
  g_kt.used = 0;
  g_kt.on = false;
  return rc;
}

static int check_ws(void* ws, size_t ws_bytes) {
  if (!ws || ((uintptr_t)ws & 255)) return CAFEQ_ERR_WORKSPACE;
  (void)ws_bytes;
  return CAFEQ_OK;
}

// The fused gradient chain reads and writes the gradient through a tensor map, which wants 16-byte alignment: a gradient array that
// starts elsewhere is filled from one in the workspace (the size queries count it).
static bool grad_off_16(const float* gradM) { return ((uintptr_t)gradM & 15) != 0; }

// Where an optimiser state keeps the inverse of the last step's transform.  The kernels move it 16 bytes at a time: one that starts
// elsewhere is copied to the workspace's own array (`ws_inv`) for the call and back.
struct StoredInverse {
  float *slot, *inv;
  long long kk;
  cudaStream_t st;
  bool copied() const { return slot && inv != slot; }
  StoredInverse(float* opt_state, float* ws_inv, long long n, bool resume, cudaStream_t stream)
      : slot(opt_state ? opt_state + CAFEQ_OPT_STATE_HEADER + 2 * n : nullptr), inv(slot && !((uintptr_t)slot & 15) ? slot : ws_inv), kk(n), st(stream) {
    if (copied() && resume) CQ_LAUNCH(copy_f32_kernel, grid_for(kk), 256, 0, st, slot, inv, kk);
  }
  void keep(int steps) const {
    if (copied() && steps > 0) CQ_LAUNCH(copy_f32_kernel, grid_for(kk), 256, 0, st, inv, slot, kk);
  }
};

static int last_launch() { return cudaGetLastError() == cudaSuccess ? CAFEQ_OK : CAFEQ_ERR_CUDA; }

// ------------------------------------------------------------------------------------------------
// Shapes whose scratch is sized for the tensor-core pass alone, so that weights which the pass cannot take (rows off 16-byte
// boundaries) are refused for lack of scratch.  A last half tile of 128 columns goes through the pass too, but its scratch stays
// that of the shape-agnostic kernels: such weights are taken at any address.
static bool sized_for_pass(const Geo& G, const void* W) {
  const bool in = G.axis == CAFEQ_AXIS_IN;
  return kk_fast(G.k) && bd_supported(in ? BD_IN : BD_OUT, G.d_out, G.d_in, G.ld, G.k, G.g, W) && (!in || G.d_in % 256 == 0);
}

// What cafeq_rtn needs from its workspace: nothing when the streaming kernel covers the call (no transform, group 32 /
// 64 / 128 / 256, aligned rows), the per-group records and the rounded operator when the fused tensor-core pass
// covers it, matrix-sized fp32 buffers otherwise.  W / codes may be null (a size query): aligned pointers are assumed.
static size_t rtn_scratch(const Geo& G, bool has_T, const void* W, const int8_t* codes, Bump* carve, MatWS* w, float** Tc) {
  Bump count(nullptr, 0);
  Bump& b = carve ? *carve : count;
  MatWS tmp;
  MatWS& m = w ? *w : tmp;
  if (!has_T && (G.g == 32 || G.g == 64 || G.g == 128 || G.g == 256) && !((uintptr_t)W & 15) && !(G.ld % 8) &&
      !((uintptr_t)codes & 7))
    return 0;
  const bool lean = has_T && sized_for_pass(G, W);
  carve_matrix(b, G, &m, false, lean);
  float* t = has_T ? b.take<float>((size_t)G.nbT * G.k * G.k) : nullptr;
  if (Tc) *Tc = t;
  return b.used;
}

extern "C" int cafeq_rtn_workspace_size(const cafeq_matrix_desc* d, int has_transform, size_t* bytes) {
  Geo G;
  int rc = make_geo(d, &G, false);
  if (rc) return rc;
  if (!bytes) return CAFEQ_ERR_INVALID_ARG;
  *bytes = rtn_scratch(G, has_transform != 0 && G.k > 0, nullptr, nullptr, nullptr, nullptr, nullptr);
  return CAFEQ_OK;
}

extern "C" int cafeq_rtn(const cafeq_matrix_desc* d, const void* W, const float* T, int8_t* codes, float* scales,
                         void* ws, size_t ws_bytes, void* stream) {
  Geo G;
  int rc = make_geo(d, &G, false);
  if (rc) return rc;
  if (!W || !codes || !scales) return CAFEQ_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const bool has_T = (T != nullptr && G.k > 0);
  if (!has_T) {
    // no transform: one streaming kernel, no scratch (the workspace may be null)
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (rtn_stream_launch(st, W, G.ld, G.d_out, G.d_in, G.g, qmax_of(d->bits), codes, scales)) return last_launch();
    g_launches.fetch_sub(1, std::memory_order_relaxed);
  }
  if ((rc = check_ws(ws, ws_bytes))) return rc;
  Bump b(ws, ws_bytes);
  MatWS w;
  float* Tc = nullptr;
  rtn_scratch(G, has_T, W, codes, &b, &w, &Tc);
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  // (other groups without a transform: one kernel from the weights themselves where rows and widths allow, the workspace unused)
  if (!has_T && launch_group_quant_vec<uint16_t>(st, (const uint16_t*)W, G.ld, G.d_out, G.ng, G.g, qmax_of(d->bits), nullptr,
                                                 CAFEQ_OFFSETS_NONE, nullptr, nullptr, nullptr, nullptr, nullptr, codes, scales, nullptr))
    return last_launch();
  forward_quant(st, W, G, d->bits, has_T ? T : nullptr, d->trole == CAFEQ_APPLY_TT, w, nullptr, CAFEQ_OFFSETS_NONE, false, nullptr, codes,
                scales, nullptr, true, nullptr, nullptr, Tc, Tc);
  return last_launch();
}

// ------------------------------------------------------------------------------------------------
// inference side: apply a block-diagonal operator to activations, dequantise packed weights
// ------------------------------------------------------------------------------------------------
static size_t apply_scratch(const Geo& G, bool fused) {
  const size_t kk = (size_t)G.nbT * G.k * G.k;
  return 1024 + kk * 6 + (fused ? 0 : (size_t)G.n * 4 + 256);
}
static Geo apply_geo(Geo G) {
  // the store epilogue ignores the quantisation groups: any group width the pass is built for will do
  if (G.d_in % 128 == 0) { G.g = 128; G.ng = G.d_in / 128; }
  return G;
}

extern "C" int cafeq_apply_workspace_size(const cafeq_matrix_desc* d, size_t* bytes) {
  Geo G;
  int rc = make_geo(d, &G, false);
  if (rc) return rc;
  if (!bytes || G.k <= 0) return CAFEQ_ERR_INVALID_ARG;
  const Geo Ga = apply_geo(G);
  // (X itself is not known here: 16-byte aligned rows are assumed; a call whose X does not qualify returns
  // CAFEQ_ERR_WORKSPACE)
  *bytes = apply_scratch(G, sized_for_pass(Ga, nullptr));
  return CAFEQ_OK;
}

extern "C" int cafeq_apply_transform(const cafeq_matrix_desc* d, const void* X, const float* T, void* Y, int32_t* status, void* ws,
                                     size_t ws_bytes, void* stream) {
  Geo G;
  int rc = make_geo(d, &G, false);
  if (rc) return rc;
  if (!X || !T || !Y || G.k <= 0) return CAFEQ_ERR_INVALID_ARG;
  if ((rc = check_ws(ws, ws_bytes))) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const long long kk = (long long)G.nbT * G.k * G.k;
  Bump b(ws, ws_bytes);
  float* Tc = b.take<float>(kk);
  uint16_t* Tb = b.take<uint16_t>(kk);
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  // the deployed operator is the bf16 rounding of the given one (what the tensor cores apply; the pass converts it
  // itself, the shape-agnostic kernels take the rounded fp32 copy)
  const int transposed = d->trole == CAFEQ_APPLY_TT;
  const long long row_groups = (G.d_out + AS_ROWS - 1) / AS_ROWS, ctas = row_groups * G.nbq * (G.k / 32);
  // Few rows: every group of eight reads the operators again, so the small kernel loses against one pass over them when groups and
  // width multiply.  Its time follows CTAs x (k + 32): 250 000 is 13 us, what the call with the pass takes on the host (two kernels
  // and a tensor map; the small kernel's 10).  Measured, small against pass, device time in us: k = 256, d_in = 8192, 24 rows
  // 12.4 / 10.1, 64 rows 26.6 / 10.3; k = 128, 14336, 24 rows 11.6 / 9.3, 64 rows 25.8 / 9.5; k = 64, 14336, 48 rows 12.7 / 8.8,
  // 64 rows 16.1 / 8.7; k = 32, 14336, 64 rows 12.2 / 8.1.  (On the device alone they meet at 108 000, 8 us.)  One group is faster at
  // every width (k = 256, 14336: 10.4 / 11.9), and what the pass does not take has only slower kernels beside this one.
  const bool few = row_groups == 1 || ctas * (G.k + 32) <= 250000 || !tc_apply_ok(G.k) || ((uintptr_t)X & 15) || G.ld % 8;
  if (G.axis == CAFEQ_AXIS_IN && few && G.d_out <= AS_MAX_ROWS && G.k % 32 == 0 && G.k <= 256 && ((uintptr_t)T & 15) == 0) {
    CQ_LAUNCH(apply_small_kernel, dim3(G.nbq * (G.k / 32), (unsigned)row_groups), 256, 0, st, (const uint16_t*)X, G.ld, T,
              reinterpret_cast<uint16_t*>(Y), G.d_out, G.d_in, G.k, G.r, transposed, status);
    return last_launch();
  }
  {
    const Geo Ga = apply_geo(G);
    BdParams p;
    memset(&p, 0, sizeof(p));
    p.epi = EPI_STORE;
    p.delta = reinterpret_cast<uint16_t*>(Y);
    if (fused_pass(st, X, G.ld, Ga, T, transposed, Tb, p, status, nullptr, Tc)) return last_launch();
  }
  float* U = b.take<float>(G.n);
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  bool applied = false;
  if (tc_apply_ok(G.k)) {
    launch_operator_bf16(st, T, Tb, G.k, G.nbT, transposed, status);
    applied = apply_tc(st, X, G, Tb, U, status);
  }
  if (!applied) {
    CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, T, Tc, kk, nullptr);
    launch_apply(st, X, 1, G.ld, G, Tc, transposed, U, G.d_in, GEMM_STORE, nullptr, status);
  }
  CQ_LAUNCH(f32_to_bf16_kernel, grid_for(G.n), 256, 0, st, U, reinterpret_cast<uint16_t*>(Y), (long long)G.n);
  return last_launch();
}

extern "C" int cafeq_dequant(const cafeq_matrix_desc* d, const uint8_t* packed, const float* scales, void* What, long long ldo,
                             void* stream) {
  Geo G;
  int rc = make_geo(d, &G, false);
  if (rc) return rc;
  if (!packed || !scales || !What || ldo < G.d_in || (G.d_in % 8)) return CAFEQ_ERR_INVALID_ARG;
  const long long n8 = G.n / 8;
  if (G.g % 8 == 0 && ldo % 8 == 0 && ((uintptr_t)What & 15) == 0 && ((uintptr_t)packed & 7) == 0 && n8 < (1ll << 31)) {
#define DQ8(B)                                                                                                           \
  case B:                                                                                                                \
    CQ_LAUNCH(dequant8_kernel<B>, (unsigned)((n8 + 1023) / 1024), 256, 0, (cudaStream_t)stream, packed, scales,          \
              reinterpret_cast<uint16_t*>(What), (unsigned)n8, (unsigned)(G.d_in / 8), (unsigned)(G.g / 8), ldo);        \
    return last_launch();
    switch (d->bits) { DQ8(2) DQ8(3) DQ8(4) DQ8(5) DQ8(6) DQ8(7) DQ8(8) }
#undef DQ8
  }
  CQ_LAUNCH(dequant_kernel, grid_for(G.n / 8), 256, 0, (cudaStream_t)stream, packed, scales, reinterpret_cast<uint16_t*>(What), G.d_out,
            G.d_in, d->bits, G.g, ldo);
  return last_launch();
}

// ------------------------------------------------------------------------------------------------
// single matrix forward + backward
// ------------------------------------------------------------------------------------------------
namespace cafeq {

struct SingleWS {
  MatWS m;
  float *Mc, *Minv, *gMinv, *tmp, *c, *A;
  double* acc;
  KkWS kk;
  // tensor-core straight-through path: second bf16 term of the residual, N = Minv^T Minv
  uint16_t* Dlo;
  float* Nf;
  bool lean;  // carved without matrix-sized scratch: only the fused surrogate path may run
  int err;    // host-side error found while enqueuing a step
};

static bool carve_single(Bump& b, const Geo& G, SingleWS* s, bool need_E, bool lean = false) {
  s->lean = lean;
  s->err = CAFEQ_OK;
  carve_matrix(b, G, &s->m, need_E, lean);
  size_t kk = (size_t)G.nbT * G.k * G.k;
  s->Mc = b.take<float>(kk);
  s->Minv = b.take<float>(kk);
  s->gMinv = b.take<float>(kk);
  s->tmp = b.take<float>(kk);
  s->c = b.take<float>((size_t)G.nbT * G.k);
  s->A = b.take<float>((size_t)G.nbT * G.k);
  s->acc = b.take<double>(8);
  carve_kk(b, G.nbT, G.k, &s->kk);
  s->Dlo = lean ? nullptr : b.take<uint16_t>(G.n);
  s->Nf = b.take<float>(kk);
  return !b.overflow;
}

// Lean workspaces: a step of Eq. 4 / LogSumExp without the quantised loss on shapes the fused pass covers leaves
// nothing matrix-sized in scratch.  (W itself is not known to the size query: 16-byte aligned rows are assumed; a
// call whose weights turn out not to qualify returns CAFEQ_ERR_WORKSPACE.)
static bool lean_single_ok(const Geo& G, const cafeq_opt_cfg* cfg, const void* W) {
  if (!cfg || cfg->loss_kind != CAFEQ_LOSS_SURROGATE || cfg->eval_every != 0) return false;
  return sized_for_pass(G, W);
}
static bool single_tc(const Geo& G) { return G.k == 32 || kk_fast(G.k); }
// Enqueue one forward(+backward) for a single matrix; gradM may be null.  hist is an optional [2] slot.  Inside a run of many steps
// (in_run, single_tc) the losses are left in s.acc for single_next_kernel, which also sets up the steps after the first (prepared).
static void single_step(cudaStream_t st, const cafeq_matrix_desc* d, const Geo& G, const void* W, const float* M,
                        float* Minv_out, const void* offsets, int off_kind, int loss_kind, float kappa, bool want_exact,
                        float* losses, float* hist, float* gradM, int32_t* status, SingleWS& s, bool force_generic,
                        bool warm = false, float* step_counter = nullptr, float* grad_offsets = nullptr, bool splits_kept = false,
                        bool in_run = false, bool prepared = false) {
  const int k = G.k;
  const bool tc = single_tc(G) && !force_generic;
  const long long kk = (long long)G.nbT * k * k;
  const float qm = qmax_of(d->bits);
  const bool ste = (loss_kind == CAFEQ_LOSS_L2_STE);
  const bool need_l2 = want_exact || ste;
  const bool want_grad = (gradM != nullptr);
  const bool in_r1 = (G.axis == CAFEQ_AXIS_IN && G.r == 1);
  // straight-through mode on the tensor cores: input axis, no rounding offsets, shapes the fused pass covers
  const bool ste_tc = ste && tc && in_r1 && off_kind == CAFEQ_OFFSETS_NONE &&
                      bd_supported(BD_IN, G.d_out, G.d_in, G.ld, k, G.g, W);
  if (tc) {
    PrepArgs pa;
    memset(&pa, 0, sizeof(pa));
    pa.M = M; pa.Mc = s.Mc; pa.Ab = s.kk.Ab; pa.kk = kk;
    pa.zero_f[0] = s.A; pa.zero_fn[0] = (long long)G.nbT * k;
    pa.zero_f[1] = s.m.agrp; pa.zero_fn[1] = G.ng;
    if (in_r1) { pa.zero_f[2] = s.m.cw; pa.zero_fn[2] = G.ng; }
    if (want_grad) { pa.zero_f[3] = gradM; pa.zero_fn[3] = kk; }
    pa.zero_d = s.acc; pa.zero_dn = in_run ? 6 : 8;
    pa.step_counter = step_counter;
    pa.step_slot = in_run ? s.acc + 6 : nullptr;
    pa.status = status;
    if (!prepared) CQ_LAUNCH(step_prep_kernel, grid_for(kk), 256, 0, st, pa);
    NsParams eq4;
    memset(&eq4, 0, sizeof(eq4));
    eq4.c = s.c;
    eq4.n = 1;
    eq4.blk0[1] = G.nbT;
    eq4.cw[0] = in_r1 ? s.m.cw : nullptr;
    eq4.g[0] = G.g;
    if ((s.err = ns_inverse(st, s.Mc, s.Minv, G.nbT, k, warm, s.kk, status, true, splits_kept && tb_supported(k, 2), &eq4))) return;
    if (!s.kk.mn) CQ_LAUNCH(colnorm_cw_kernel, dim3(k / 32, G.nbT), dim3(32, 8), 0, st, s.Minv, k, s.c, in_r1 ? s.m.cw : nullptr, G.g);
    if (!in_r1) {
      if (G.axis == CAFEQ_AXIS_IN) CQ_LAUNCH(cw_in_kernel, (G.ng + 127) / 128, 128, 0, st, s.c, G.d_in, G.g, k, G.r, s.m.cw);
      else CQ_LAUNCH(cw_out_kernel, (G.d_out + 127) / 128, 128, 0, st, s.c, G.d_out, G.g, k, G.r, s.m.cw);
    }
  } else {
    CQ_LAUNCH(zero_f64_kernel, 1, 32, 0, st, s.acc, 8);
    CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, M, s.Mc, kk, status);
    if (step_counter) CQ_LAUNCH(adam_tick_kernel, 1, 1, 0, st, step_counter, status);
    launch_inverse(st, s.Mc, s.Minv, s.c, G.nbT, k, status);
    if (G.axis == CAFEQ_AXIS_IN) CQ_LAUNCH(cw_in_kernel, (G.ng + 127) / 128, 128, 0, st, s.c, G.d_in, G.g, k, G.r, s.m.cw);
    else CQ_LAUNCH(cw_out_kernel, (G.d_out + 127) / 128, 128, 0, st, s.c, G.d_out, G.g, k, G.r, s.m.cw);
    CQ_LAUNCH(fill_f32_kernel, grid_for(G.nbT * k), 256, 0, st, s.A, 0.f, (long long)G.nbT * k);
    CQ_LAUNCH(fill_f32_kernel, grid_for(G.ng), 256, 0, st, s.m.agrp, 0.f, G.ng);
    if (want_grad) CQ_LAUNCH(fill_f32_kernel, grid_for(kk), 256, 0, st, gradM, 0.f, kk);
  }
  if (Minv_out && Minv_out != s.Minv) CQ_LAUNCH(copy_f32_kernel, grid_for(kk), 256, 0, st, s.Minv, Minv_out, kk);
  BdParams sp;
  memset(&sp, 0, sizeof(sp));
  sp.cw = s.m.cw;
  sp.kappa = kappa;
  sp.coef = (want_grad && !ste) ? s.m.coef : nullptr;
  sp.lossacc = s.acc + 0;
  sp.Aacc = (G.axis == CAFEQ_AXIS_IN) ? s.m.agrp : s.A;
  if (ste_tc) {
    sp.delta_lo = s.Dlo;
    sp.a_always = 1;
  }
  if (s.lean && (ste || need_l2 || !tc || force_generic || off_kind != CAFEQ_OFFSETS_NONE ||
                 !bd_supported(G.axis == CAFEQ_AXIS_IN ? BD_IN : BD_OUT, G.d_out, G.d_in, G.ld, k, G.g, W))) {
    s.err = CAFEQ_ERR_WORKSPACE;  // this mode needs the matrix-sized scratch the workspace was sized without
    return;
  }
  const bool fused = forward_quant(st, W, G, d->bits, s.Mc, 0, s.m, offsets, off_kind, need_l2, nullptr, nullptr, nullptr,
                                   status, (!ste || ste_tc) && !force_generic, &sp, tc ? s.kk.Ab : nullptr, nullptr, s.tmp);
  if (ste_tc && fused) {
    // Nothing below needs E = Minv o Delta itself.  With Gram_B = sum_o Delta[o, B]^T Delta[o, B] (k x k per block) and
    // N = Minv^T Minv:  L2 = <N, Gram>,  dL/dMinv = 2 Minv Gram,  gDelta = 2 N o Delta (one more block-diagonal
    // apply), and the scale path needs sum_e gDelta_e Delta_e per group.  Every product runs on the tensor cores
    // with the residual as a two-term bf16 split (three-term products: fp32-grade).
    KkWS& w = s.kk;
    if (split_wanted(k, G.d_out, G.nbT, 1)) {  // Gram (fp32 in s.tmp, splits in w.Ph / w.Pl): contraction over the rows of the residual as it is stored
      const TgOperand o[2] = {TgOperand{s.m.Dbf, G.d_out, G.d_in, G.d_in}, TgOperand{s.Dlo, G.d_out, G.d_in, G.d_in}};
      if ((s.err = launch_split_product(st, 2, o, 2, o, G.d_out, G.nbT, 1, 1, s.m.D, s.tmp, w.Ph, w.Pl, status))) return;
    } else {
      TgOperand oa[3], ob[3];
      const uint16_t* at[3] = {s.m.Dbf, s.Dlo, s.m.Dbf};
      const uint16_t* bt[3] = {s.m.Dbf, s.m.Dbf, s.Dlo};
      for (int t = 0; t < 3; ++t) {
        oa[t] = TgOperand{at[t], G.d_out, G.d_in, G.d_in};
        ob[t] = TgOperand{bt[t], G.d_out, G.d_in, G.d_in};
      }
      TgParams p;
      memset(&p, 0, sizeof(p));
      p.M = p.N = k; p.K = (G.d_out + 63) / 64 * 64; p.batch = G.nbT; p.nterms = 3;  // (rows past the end read as zeros)
      p.a_mn = p.b_mn = 1;
      p.colsA_per_batch = p.colsB_per_batch = k;
      p.divA = 1;
      p.alpha = 1.f;
      p.C = s.tmp; p.ldc = k; p.sCb = (long long)k * k;
      p.Chi = w.Ph; p.Clo = w.Pl;
      p.min_ctas = 148;  // a long contraction: as many CTAs as the tile shapes give
      p.status = status;
      g_launches.fetch_add(1, std::memory_order_relaxed);
      if ((s.err = tg_launch(st, oa, ob, p))) return;
    }
    {  // N = Minv^T Minv (fp32 in s.Nf, splits in w.Qh / w.Ql)
      if (w.mn) {  // both operands are X read transposed from its row-major splits
        const uint16_t* a1[3] = {w.Xh, w.Xl, w.Xh};
        const uint16_t* b1[3] = {w.Xh, w.Xh, w.Xl};
        s.err = launch_kk_tc(st, 3, a1, b1, G.nbT, k, 1.f, 0.f, 0.f, nullptr, s.Nf, w.Qh, w.Ql, nullptr, nullptr, nullptr, status, 1, 1, 1);
      } else {
        const uint16_t* a1[3] = {w.XTh, w.XTl, w.XTh};
        const uint16_t* b1[3] = {w.XTh, w.XTh, w.XTl};
        s.err = launch_kk_tc(st, 3, a1, b1, G.nbT, k, 1.f, 0.f, 0.f, nullptr, s.Nf, w.Qh, w.Ql, nullptr, nullptr, nullptr, status);
      }
      if (s.err) return;
    }
    CQ_LAUNCH(dot_f32_kernel, grid_for(kk), 256, 0, st, s.Nf, s.tmp, kk, s.acc + 1);
    CQ_LAUNCH(sqsum_bf16_kernel, grid_for(G.n), 256, 0, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, s.acc + 2, status);
    if (!in_run) CQ_LAUNCH(finalize_single_kernel, 1, 1, 0, st, s.acc, losses, hist, 1);
    if (!want_grad) return;
    {  // dL/dMinv = 2 Minv Gram (Gram is symmetric: its rows serve as the contraction-major second operand)
      const uint16_t* a2[3] = {w.Xh, w.Xl, w.Xh};
      const uint16_t* b2[3] = {w.Ph, w.Ph, w.Pl};
      if ((s.err = launch_kk_tc(st, 3, a2, b2, G.nbT, k, 2.f, 0.f, 0.f, nullptr, s.gMinv, nullptr, nullptr, nullptr, nullptr, nullptr,
                   status))) return;
    }
    // gDelta[o, B k + j] = 2 sum_l N_B[j][l] Delta[o, B k + l], and per group the sum of gDelta Delta.  Blocks of 256 from 2^21 entries
    // on: as the product's epilogue (256 x 512 188.8 -> 193.0 us a call, 1024 x 1024 206.8 -> 209.0, 4096 x 512 206.6 -> 206.4,
    // 1500 x 2048 219 -> 212, 4096 x 3584 328 -> 312).
    if (k == 256 && G.n >= 1ll << 21) {
      const T2Ste ste{s.m.Dbf, s.Dlo, G.d_in, s.m.a, s.m.usel, s.m.coef, G.g};
      g_launches.fetch_add(1, std::memory_order_relaxed);
      if ((s.err = tg_launch_ste(st, w.Qh, w.Ql, G.d_out, G.nbT, 2.f, ste, status))) return;
    } else {  // gDelta in s.m.D (fp32 [d_out, d_in])
      TgOperand oa[3], ob[3];
      const uint16_t* at[3] = {s.m.Dbf, s.Dlo, s.m.Dbf};
      const uint16_t* bt[3] = {w.Qh, w.Qh, w.Ql};
      for (int t = 0; t < 3; ++t) {
        oa[t] = TgOperand{at[t], G.d_out, G.d_in, G.d_in};
        ob[t] = TgOperand{bt[t], (long long)G.nbT * k, k, k};
      }
      TgParams p;
      memset(&p, 0, sizeof(p));
      p.M = G.d_out; p.N = k; p.K = k; p.batch = G.nbT; p.nterms = 3;
      p.rowsA_per_batch = 0; p.colsA_per_batch = k; p.rowsB_per_batch = k;
      p.divA = 1;
      p.alpha = 2.f;
      p.C = s.m.D; p.ldc = G.d_in; p.sCb = k;  // batch b writes the columns [b k, b k + k)
      p.status = status;
      g_launches.fetch_add(1, std::memory_order_relaxed);
      if ((s.err = tg_launch(st, oa, ob, p))) return;
      const long long nrec = (long long)G.d_out * G.ng;
      CQ_LAUNCH(ste_scale_coef_kernel, (unsigned)((nrec * 32 + 255) / 256), 256, 0, st, s.m.D, (long long)G.d_in, s.m.Dbf, s.Dlo,
                (long long)G.d_in, G.d_out, G.ng, G.g, s.m.a, s.m.usel, 1, s.m.coef, status);
    }
    launch_scatter(st, W, G, s.m.coef, s.m.idx, gradM, 0, status, 1);
    s.err = minv_path_tc(st, s.Minv, s.gMinv, gradM, G.nbT, k, s.kk, status);
    return;
  }
  if (need_l2) {
    // E = Minv o Delta, L2 = sum E^2
    bool done = false;
    if (fused) {
      BdParams bp;
      memset(&bp, 0, sizeof(bp));
      bp.epi = EPI_SQSUM;
      bp.sqacc = s.acc + 1;
      done = fused_pass(st, s.m.Dbf, G.d_in, G, s.Minv, 0, s.m.Tb, bp, status, nullptr, s.tmp);
    }
    if (!done)
      launch_apply(st, s.m.D, 0, G.d_in, G, s.Minv, 0, s.m.E, G.d_in, (ste ? GEMM_STORE : 0) | GEMM_SQSUM, s.acc + 1, status);
    CQ_LAUNCH(sqsum_bf16_kernel, grid_for(G.n), 256, 0, st, (const uint16_t*)W, G.ld, G.d_out, G.d_in, s.acc + 2, status);
  }
  if (!fused)
    CQ_LAUNCH(surrogate_rows_kernel, (G.d_out + 127) / 128, 128, 0, st, s.m.a, s.m.usel, G.d_out, G.ng, G.g, G.axis,
                                                                 s.m.cw, kappa, k, G.r, (want_grad && !ste) ? s.m.coef : nullptr,
                                                                 s.m.agrp, s.A, s.acc + 0, status);
  if (G.axis == CAFEQ_AXIS_IN && !in_r1)
    CQ_LAUNCH(expand_agrp_kernel, (G.d_in + 127) / 128, 128, 0, st, s.m.agrp, G.d_in, G.g, k, G.r, s.A);
  if (!in_run) CQ_LAUNCH(finalize_single_kernel, 1, 1, 0, st, s.acc, losses, hist, need_l2 ? 1 : 0);
  if (!want_grad) return;
  if (!ste) {
    launch_scatter(st, W, G, s.m.coef, s.m.idx, gradM, 0, status, fused ? 1 : 0);
    if (tc) {
      ChainParams cp;
      memset(&cp, 0, sizeof(cp));
      cp.n = 1;
      cp.blk0[1] = G.nbT;
      cp.A[0] = s.A; cp.Agrp[0] = in_r1 ? s.m.agrp : nullptr; cp.g[0] = G.g; cp.scale[0] = 2.f * kappa;
      cp.X = s.Minv;
      s.err = minv_path_tc(st, s.Minv, nullptr, gradM, G.nbT, k, s.kk, status, &cp);
      return;
    }
    CQ_LAUNCH(gminv_kernel, grid_for(kk), 256, 0, st, s.Minv, s.A, in_r1 ? s.m.agrp : nullptr, G.g, 2.f * kappa, k, kk, s.gMinv);
  } else {
    // gMinv = 2 * sum_free E Delta^T ; gDelta = 2 Minv^T o E (overwrites Delta) ; scale path through arg-max
    CQ_LAUNCH(fill_f32_kernel, grid_for(kk), 256, 0, st, s.gMinv, 0.f, kk);
    launch_opgrad(st, s.m.E, G.d_in, s.m.D, 0, G.d_in, G, s.gMinv, 0, 2.f, status);
    launch_apply(st, s.m.E, 0, G.d_in, G, s.Minv, 1, s.m.D, G.d_in, GEMM_STORE, nullptr, status, 2.f);
    if (grad_offsets)  // s.m.D holds d L2 / d Uhat = 2 Minv^T E
      CQ_LAUNCH(grad_offsets_kernel, grid_for(G.n), 256, 0, st, s.m.U, s.m.D, (long long)G.d_in, G.d_out, G.d_in, G.g, s.m.a, qm,
                grad_offsets, status);
    CQ_LAUNCH(ste_scale_path_kernel, (unsigned)(((long long)G.d_out * G.ng * 32 + 255) / 256), 256, 0, st, 
        s.m.U, s.m.D, G.d_in, G.d_out, G.ng, G.g, s.m.a, s.m.usel, qm, offsets, off_kind, G.d_in, s.m.coef, status);
    launch_scatter(st, W, G, s.m.coef, s.m.idx, gradM, 0, status, 0);
  }
  // gradM -= Minv^T gMinv Minv^T
  if (tc) {
    s.err = minv_path_tc(st, s.Minv, s.gMinv, gradM, G.nbT, k, s.kk, status);
  } else {
    launch_kk(st, s.Minv, 1, s.gMinv, 0, s.tmp, G.nbT, k, 1.f, GEMM_STORE, status);
    launch_kk(st, s.tmp, 0, s.Minv, 1, gradM, G.nbT, k, -1.f, GEMM_STORE | GEMM_ACCUM, status);
  }
}

}  // namespace cafeq

extern "C" int cafeq_proxy_loss_fwd_bwd(const cafeq_matrix_desc* d, const void* W, const float* M, float* Minv,
                                        const void* offsets, int offsets_kind, int loss_kind, float kappa, int flags,
                                        float* losses, float* gradM, float* grad_offsets, int32_t* status, void* ws,
                                        size_t ws_bytes, void* stream) {
  Geo G;
  int rc = make_geo(d, &G, true);
  if (rc) return rc;
  if (!W || !M || !losses) return CAFEQ_ERR_INVALID_ARG;
  // the gradient with respect to soft offsets belongs to the straight-through loss evaluated with soft offsets
  if (grad_offsets && (offsets_kind != CAFEQ_OFFSETS_SOFT_F32 || loss_kind != CAFEQ_LOSS_L2_STE || (flags & CAFEQ_FLAG_NO_GRAD)))
    return CAFEQ_ERR_INVALID_ARG;
  if (loss_kind != CAFEQ_LOSS_SURROGATE && loss_kind != CAFEQ_LOSS_L2_STE) return CAFEQ_ERR_INVALID_ARG;
  if (offsets_kind < CAFEQ_OFFSETS_NONE || offsets_kind > CAFEQ_OFFSETS_SOFT_F32) return CAFEQ_ERR_INVALID_ARG;
  if (offsets_kind != CAFEQ_OFFSETS_NONE && !offsets) return CAFEQ_ERR_INVALID_ARG;
  const bool want_grad = !(flags & CAFEQ_FLAG_NO_GRAD);
  if (want_grad && !gradM) return CAFEQ_ERR_INVALID_ARG;
  if ((rc = check_ws(ws, ws_bytes))) return rc;
  if (kappa <= 0.f) kappa = 1.f / (float)(((1 << d->bits) - 1) * ((1 << d->bits) - 1));
  cudaStream_t st = (cudaStream_t)stream;
  Bump b(ws, ws_bytes);
  SingleWS s;
  const long long kk = (long long)G.nbT * G.k * G.k;
  const bool off_grad = want_grad && grad_off_16(gradM);
  // Eq. 4 alone on a shape the tensor-core pass covers leaves nothing matrix-sized in scratch (the lean size of
  // cafeq_workspace_size with a CAFEQ_LOSS_SURROGATE configuration is enough); everything else takes the full carving
  bool lean = false;
  if (loss_kind == CAFEQ_LOSS_SURROGATE && !(flags & (CAFEQ_FLAG_EXACT_LOSS | CAFEQ_FLAG_GENERIC)) &&
      offsets_kind == CAFEQ_OFFSETS_NONE) {
    cafeq_opt_cfg c0;
    memset(&c0, 0, sizeof(c0));
    c0.loss_kind = CAFEQ_LOSS_SURROGATE;
    lean = lean_single_ok(G, &c0, W);
    if (lean) {  // a workspace that holds the full carving keeps using it
      Bump probe(nullptr, 0);
      SingleWS tmp;
      carve_single(probe, G, &tmp, true, false);
      if (off_grad) probe.take<float>(kk);
      if (probe.used <= ws_bytes) lean = false;
    }
  }
  if (!carve_single(b, G, &s, true, lean)) return CAFEQ_ERR_WORKSPACE;
  float* grad = off_grad ? b.take<float>(kk) : gradM;
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  const bool warm = (flags & CAFEQ_FLAG_WARM_MINV) && Minv;
  if (warm) CQ_LAUNCH(copy_f32_kernel, grid_for(kk), 256, 0, st, Minv, s.Minv, kk);
  single_step(st, d, G, W, M, Minv, offsets, offsets_kind, loss_kind, kappa, (flags & CAFEQ_FLAG_EXACT_LOSS) != 0, losses,
              nullptr, want_grad ? grad : nullptr, status, s, (flags & CAFEQ_FLAG_GENERIC) != 0, warm, nullptr, grad_offsets);
  if (s.err) return s.err;
  if (off_grad) CQ_LAUNCH(copy_f32_kernel, grid_for(kk), 256, 0, st, grad, gradM, kk);
  return last_launch();
}

extern "C" int cafeq_optimize_single(const cafeq_matrix_desc* d, const void* W, float* M, float* opt_state,
                                     const cafeq_opt_cfg* cfg, float* loss_history, int32_t* status, void* ws,
                                     size_t ws_bytes, void* stream) {
  Geo G;
  int rc = make_geo(d, &G, true);
  if (rc) return rc;
  if (!W || !M || !cfg || cfg->struct_size != sizeof(cafeq_opt_cfg) || !loss_history) return CAFEQ_ERR_INVALID_ARG;
  if (cfg->steps < 0) return CAFEQ_ERR_INVALID_ARG;
  if (cfg->loss_kind != CAFEQ_LOSS_SURROGATE && cfg->loss_kind != CAFEQ_LOSS_L2_STE) return CAFEQ_ERR_INVALID_ARG;
  if (cfg->optimizer == CAFEQ_OPT_ADAM && !opt_state) return CAFEQ_ERR_INVALID_ARG;
  if (cfg->optimizer != CAFEQ_OPT_ADAM && cfg->optimizer != CAFEQ_OPT_GD) return CAFEQ_ERR_INVALID_ARG;
  if ((rc = check_ws(ws, ws_bytes))) return rc;
  float kappa = cfg->kappa;
  if (kappa <= 0.f) kappa = 1.f / (float)(((1 << d->bits) - 1) * ((1 << d->bits) - 1));
  cudaStream_t st = (cudaStream_t)stream;
  Bump b(ws, ws_bytes);
  SingleWS s;
  if (!carve_single(b, G, &s, true, lean_single_ok(G, cfg, W))) return CAFEQ_ERR_WORKSPACE;
  const long long kk = (long long)G.nbT * G.k * G.k;
  float* grad = b.take<float>(kk);
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  // the inverse of the last step's transform lives in the optimiser state, so a resumed run refines it
  const bool resume = cfg->resume && opt_state;
  const StoredInverse stored(opt_state, s.Minv, kk, resume, st);
  s.Minv = stored.inv;
  for (int it = 0; it < cfg->steps; ++it) {
    bool eval = cfg->eval_every > 0 && (it % cfg->eval_every == 0);
    const bool in_run = single_tc(G);
    single_step(st, d, G, W, M, nullptr, nullptr, CAFEQ_OFFSETS_NONE, cfg->loss_kind, kappa, eval, nullptr,
                loss_history + 2 * (size_t)it, grad, status, s, false, resume || it > 0, opt_state, nullptr, it > 0, in_run,
                in_run && it > 0);
    if (s.err) return s.err;
    if (in_run) {
      SingleNextArgs na;
      memset(&na, 0, sizeof(na));
      na.M = M; na.grad = grad; na.state = opt_state; na.kk = kk;
      na.adam = cfg->optimizer == CAFEQ_OPT_ADAM;
      na.lr = cfg->lr; na.b1 = cfg->beta1; na.b2 = cfg->beta2; na.eps = cfg->eps;
      na.acc = s.acc; na.hist = loss_history + 2 * (size_t)it;
      na.want_exact = eval || cfg->loss_kind == CAFEQ_LOSS_L2_STE;
      na.next = it + 1 < cfg->steps; na.slot = 6 + (it & 1);
      na.Mc = s.Mc; na.Ab = s.kk.Ab;
      na.zero_f[0] = s.A; na.zero_fn[0] = (long long)G.nbT * G.k;
      na.zero_f[1] = s.m.agrp; na.zero_fn[1] = G.ng;
      if (G.axis == CAFEQ_AXIS_IN && G.r == 1) { na.zero_f[2] = s.m.cw; na.zero_fn[2] = G.ng; }
      na.status = status;
      CQ_LAUNCH(single_next_kernel, grid_for(kk), 256, 0, st, na);
    } else if (cfg->optimizer == CAFEQ_OPT_GD) {
      CQ_LAUNCH(gd_update_kernel, grid_for(kk), 256, 0, st, M, grad, cfg->lr, kk, status);
    } else {
      CQ_LAUNCH(adam_update_kernel, grid_for(kk), 256, 0, st, M, grad, opt_state, cfg->lr, cfg->beta1, cfg->beta2, cfg->eps, kk,
                                                       status);
    }
  }
  stored.keep(cfg->steps);
  return last_launch();
}

// ------------------------------------------------------------------------------------------------
// pair
// ------------------------------------------------------------------------------------------------
namespace cafeq {

static int make_pair_geo(const cafeq_matrix_desc* d1, const cafeq_matrix_desc* d2, Geo* G1, Geo* G2) {
  int rc = make_geo(d1, G1, true);
  if (rc) return rc;
  if ((rc = make_geo(d2, G2, true))) return rc;
  if (G1->axis != CAFEQ_AXIS_OUT || G2->axis != CAFEQ_AXIS_IN) return CAFEQ_ERR_INVALID_ARG;
  if (G1->k != G2->k || G1->r != 1) return CAFEQ_ERR_INVALID_ARG;
  if (G1->nbT != G2->nbT) return CAFEQ_ERR_INVALID_ARG;  // h / k operator blocks on both sides
  if (d1->bits != d2->bits) return CAFEQ_ERR_UNSUPPORTED;
  return CAFEQ_OK;
}

// Cm[x][y] = sum over blocks B of W2:  A1[(B/r)k + j][x] * A2[y][B k + j]   (A1 stored [h, d1], A2 stored [d3, r h])
static void launch_pair_product(cudaStream_t st, const void* A1, int a1_bf16, long long ld1, const void* A2, int a2_bf16,
                                long long ld2, const Geo& G1, const Geo& G2, float* Cm, const int32_t* status) {
  const int d1n = G1.d_in, d3n = G2.d_out, k = G1.k;
  GemmArgs g = gemm_defaults(status);
  g.M = d1n; g.N = d3n;
  g.A = A1; g.a_bf16 = a1_bf16; g.sAm = 1; g.sAk = ld1;
  g.B = A2; g.b_bf16 = a2_bf16; g.sBk = 1; g.sBn = ld2;
  g.C = Cm; g.sCm = d3n; g.sCn = 1; g.sCb = 0;
  if (G2.r == 1) {
    g.K = G1.d_out; g.batch = 1;
    g.mode = GEMM_STORE;
  } else {
    CQ_LAUNCH(fill_f32_kernel, grid_for((long long)d1n * d3n), 256, 0, st, Cm, 0.f, (long long)d1n * d3n);
    g.K = k; g.batch = G2.nbq;
    g.sAb = (long long)k * ld1; g.divA = G2.r;
    g.sBb = k;
    g.mode = GEMM_STORE | GEMM_ATOMIC;
  }
  launch_gemm(st, g);
}

struct PairWS {
  MatWS m1, m2;
  float *Mc, *Minv, *Minv_c, *gMinv, *tmp, *RM, *amax, *R;
  float *G1, *G2, *T1, *T2;  // Appendix D.1's weighted objective: block Grams of the two weights, G1 Mc, Minv_c G2
  double* acc;
  KkWS kk;
  DenseWS dn;
  bool dense;  // the product term runs on the tensor cores (every dimension a multiple of 64)
  uint16_t *gVh, *gVl;          // [d3, r h]: split of the second factor's gradient
  bool lean;                    // carved without matrix-sized scratch: only the fused LogSumExp path may run
  int err;
};

// Operator gradients of a block-diagonal apply as batched k x k tensor-core products with a two-term split of the fp32 factor.
// Output axis: out[b][m][n] = sum_l A[b k + m][l] (Bh + Bl)[b k + n][l]; A bf16 [nb k, K] (pitch lda), Bh / Bl [nb k, K].
// parts: scratch of nb k K floats.
static int opgrad_out_tc(cudaStream_t st, const uint16_t* A, long long lda, const uint16_t* Bh, const uint16_t* Bl, int nb, int k, int K,
                         float* parts, float* out, int32_t* status) {
  TgOperand oa[2], ob[2];
  if (split_wanted(k, K, nb, 1)) {
    oa[0] = TgOperand{A, (long long)nb * k, K, lda};
    ob[0] = TgOperand{Bh, (long long)nb * k, K, K};
    ob[1] = TgOperand{Bl, (long long)nb * k, K, K};
    return launch_split_product(st, 1, oa, 2, ob, K, nb, 1, 0, parts, out, nullptr, nullptr, status);
  }
  oa[0] = oa[1] = TgOperand{A, (long long)nb * k, K, lda};
  ob[0] = TgOperand{Bl, (long long)nb * k, K, K};
  ob[1] = TgOperand{Bh, (long long)nb * k, K, K};
  TgParams p;
  memset(&p, 0, sizeof(p));
  p.M = p.N = k; p.K = K; p.batch = nb; p.nterms = 2;
  p.rowsA_per_batch = p.rowsB_per_batch = k;
  p.divA = 1;
  p.alpha = 1.f;
  p.C = out; p.ldc = k; p.sCb = (long long)k * k;
  p.min_ctas = 148;  // long contraction, few output tiles: the narrowest tile
  p.status = status;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return tg_launch(st, oa, ob, p);
}
// Input axis: out[b][m][n] = sum over replicas and rows o of (Ah + Al)[o][(b r + rep) k + m] B[o][(b r + rep) k + n]; both
// factors as they are stored (contraction down the rows: MN-major operands), B bf16 [R, nb r k] (pitch ldb), Ah / Al dense.  parts: scratch
// of R nb r k floats.
static int opgrad_in_tc(cudaStream_t st, const uint16_t* Ah, const uint16_t* Al, const uint16_t* B, long long ldb, int nb, int r, int k,
                        int R, float* parts, float* out, int32_t* status) {
  if (split_wanted(k, R, nb, r)) {
    const long long all = (long long)nb * r * k;
    const TgOperand a[2] = {TgOperand{Ah, R, all, all}, TgOperand{Al, R, all, all}}, b = TgOperand{B, R, all, ldb};
    return launch_split_product(st, 2, a, 1, &b, R, nb, r, 1, parts, out, nullptr, nullptr, status);
  }
  for (int rep = 0; rep < r; ++rep) {
    TgOperand oa[2], ob[2];
    const long long cols = (long long)nb * r * k, c0 = (long long)rep * k;
    oa[0] = TgOperand{Al + c0, R, cols - c0, cols};
    oa[1] = TgOperand{Ah + c0, R, cols - c0, cols};
    ob[0] = ob[1] = TgOperand{B + c0, R, cols - c0, ldb};
    TgParams p;
    memset(&p, 0, sizeof(p));
    p.M = p.N = k; p.K = R; p.batch = nb; p.nterms = 2;
    p.a_mn = p.b_mn = 1;
    p.colsA_per_batch = p.colsB_per_batch = r * k;
    p.divA = 1;
    p.alpha = 1.f;
    p.beta = rep ? 1.f : 0.f;
    p.C0 = rep ? out : nullptr; p.ldc0 = k; p.sC0b = (long long)k * k;
    p.C = out; p.ldc = k; p.sCb = (long long)k * k;
    p.min_ctas = 148;
    p.status = status;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    const int rc = tg_launch(st, oa, ob, p);
    if (rc) return rc;
  }
  return CAFEQ_OK;
}

// straight-through gradient of one factor as operand splits (ste_grad_split_kernel); gX has one column per r replicas
static bool ste_split_ok(int g) { return g % 4 == 0 && g <= 1024; }
static void launch_ste_split(cudaStream_t st, const MatWS& m, const float* gX, long long ldg, const Geo& G, int k, int r, float qmax,
                             uint16_t* hi, uint16_t* lo, int32_t* status) {
  const long long groups = (long long)G.d_out * G.ng;
#define SGS(L, N)                                                                                                              \
  CQ_LAUNCH((ste_grad_split_kernel<L, N>), (unsigned)((groups * L + 255) / 256), 256, 0, st, m.U, gX, ldg, G.d_out, G.ng, G.g, k, r, \
            m.a, m.usel, m.idx, qmax, hi, lo, status)
  const bool few = groups * G.g < 1ll << 20;  // (as in launch_group_quant_vec)
  if (few && G.g <= 32) SGS(8, 1);
  else if (few && G.g <= 64) SGS(16, 1);
  else if (few && G.g <= 128) SGS(32, 1);
  else if (few && G.g <= 256) SGS(32, 2);
  else if (G.g <= 32) SGS(4, 2);
  else if (G.g <= 64) SGS(4, 4);
  else if (G.g <= 128) SGS(8, 4);
  else if (G.g <= 256) SGS(16, 4);
  else if (G.g <= 512) SGS(32, 4);
  else SGS(32, 8);
#undef SGS
}

static bool dense_ok(const Geo& G1, const Geo& G2) {
  return G1.d_out % 64 == 0 && G1.d_in % 64 == 0 && G2.d_out % 64 == 0 && G2.d_in % 64 == 0 && G1.k % 32 == 0;
}

static bool carve_pair(Bump& b, const Geo& G1, const Geo& G2, PairWS* p, bool need_R, bool lean = false) {
  p->lean = lean;
  p->err = CAFEQ_OK;
  carve_matrix(b, G1, &p->m1, true, lean);
  carve_matrix(b, G2, &p->m2, true, lean);
  size_t kk = (size_t)G1.nbT * G1.k * G1.k;
  p->Mc = b.take<float>(kk);
  p->Minv = b.take<float>(kk);
  p->Minv_c = b.take<float>(kk);
  p->gMinv = b.take<float>(kk);
  p->tmp = b.take<float>(kk);
  p->RM = b.take<float>(kk);
  p->G1 = b.take<float>(kk); p->G2 = b.take<float>(kk); p->T1 = b.take<float>(kk); p->T2 = b.take<float>(kk);
  p->amax = b.take<float>(64);
  p->acc = b.take<double>(8);
  p->R = need_R ? b.take<float>((size_t)G1.d_in * G2.d_out) : nullptr;
  carve_kk(b, G1.nbT, G1.k, &p->kk);
  p->dense = need_R && dense_ok(G1, G2);
  if (p->dense) carve_dense(b, G1.d_out, G1.d_in, G2.d_out, G2.r, G1.k, G1.ng, G2.ng, &p->dn);
  p->gVh = p->gVl = nullptr;
  if (p->dense) {
    p->gVh = b.take<uint16_t>(G2.n);
    p->gVl = b.take<uint16_t>(G2.n);
  }
  return !b.overflow;
}

static bool lean_pair_ok(const Geo& G1, const Geo& G2, const cafeq_opt_cfg* cfg, const void* W1, const void* W2) {
  if (!cfg || cfg->eval_every != 0) return false;
  if (cfg->loss_kind != CAFEQ_LOSS_LSE && cfg->loss_kind != CAFEQ_LOSS_SUMSQ && cfg->loss_kind != CAFEQ_LOSS_SUMSQ_WEIGHTED) return false;
  return sized_for_pass(G1, W1) && sized_for_pass(G2, W2);
}

// Block Grams of a pair's weights (constants of a run): G1[b][i][j] = sum_x W1[b k + i, x] W1[b k + j, x] and
// G2[b][i][j] = sum over the r replicas and the rows y of W2[y, (b r + rep) k + i] W2[y, (b r + rep) k + j].
static void pair_grams(cudaStream_t st, const void* W1, const Geo& G1, const void* W2, const Geo& G2, PairWS& p, const int32_t* status) {
  const int k = G1.k;
  const long long kk = (long long)G1.nbT * k * k;
  GemmArgs g = gemm_defaults(status);
  g.M = k; g.N = k; g.K = G1.d_in; g.batch = G1.nbT;
  g.A = W1; g.a_bf16 = 1; g.sAm = G1.ld; g.sAk = 1; g.sAb = (long long)k * G1.ld;
  g.B = W1; g.b_bf16 = 1; g.sBk = 1; g.sBn = G1.ld; g.sBb = (long long)k * G1.ld;
  g.C = p.G1; g.sCm = k; g.sCn = 1; g.sCb = (long long)k * k;
  g.mode = GEMM_STORE;
  launch_gemm(st, g);
  CQ_LAUNCH(fill_f32_kernel, grid_for(kk), 256, 0, st, p.G2, 0.f, kk);
  GemmArgs h = gemm_defaults(status);
  h.M = k; h.N = k; h.K = G2.d_out; h.batch = G2.nbq;
  h.A = W2; h.a_bf16 = 1; h.sAm = 1; h.sAk = G2.ld; h.sAb = k;
  h.B = W2; h.b_bf16 = 1; h.sBk = G2.ld; h.sBn = 1; h.sBb = k;
  h.C = p.G2; h.sCm = k; h.sCn = 1; h.sCb = (long long)k * k; h.divC = G2.r;
  h.mode = GEMM_STORE | GEMM_ATOMIC;
  launch_gemm(st, h);
}

// One Cayley step on the rotations (Appendix D.2's strictly orthonormal baseline): V <- beta V + g,
// A = V M^T - M V^T, M <- (I + lr/2 A)^-1 (I - lr/2 A) M, the solve by the fixed-point iteration
// Y <- M - lr/2 A (M + Y) from Y = M - lr A M (five rounds: the error falls by lr/2 ||A|| per round).
static void cayley_update(cudaStream_t st, float* M, const float* grad, float* V, float lr, float beta, int nb, int k, PairWS& p,
                          const int32_t* status) {
  const long long kk = (long long)nb * k * k;
  float *A = p.tmp, *Y = p.RM, *S = p.gMinv, *Pm = p.Minv_c;
  CQ_LAUNCH(momentum_kernel, grid_for(kk), 256, 0, st, V, beta, grad, kk, status);
  launch_kk(st, V, 0, M, 1, S, nb, k, 1.f, GEMM_STORE, status);            // V M^T
  CQ_LAUNCH(skew_blocks_kernel, grid_for(kk), 256, 0, st, S, A, k, kk);    // A = V M^T - M V^T
  launch_kk(st, A, 0, M, 0, Pm, nb, k, 1.f, GEMM_STORE, status);
  CQ_LAUNCH(lincomb_kernel, grid_for(kk), 256, 0, st, Y, M, -lr, Pm, kk, status);
  for (int it = 0; it < 5; ++it) {
    CQ_LAUNCH(lincomb_kernel, grid_for(kk), 256, 0, st, S, M, 1.f, Y, kk, status);
    launch_kk(st, A, 0, S, 0, Pm, nb, k, 1.f, GEMM_STORE, status);
    CQ_LAUNCH(lincomb_kernel, grid_for(kk), 256, 0, st, Y, M, -0.5f * lr, Pm, kk, status);
  }
  CQ_LAUNCH(copy_f32_kernel, grid_for(kk), 256, 0, st, Y, M, kk);
}

static void pair_step(cudaStream_t st, const cafeq_matrix_desc* d1, const cafeq_matrix_desc* d2, const Geo& G1, const Geo& G2,
                      const void* W1, const void* W2, const float* M, const float* P, float t, float lambda, bool want_pqe,
                      float* losses, float* hist, float* gradM, int32_t* status, PairWS& p, bool force_generic,
                      bool warm = false, float* step_counter = nullptr, bool ste = false, int objective = 0, bool splits_kept = false) {
  const int k = G1.k;
  const bool tc = kk_fast(k) && !force_generic;
  const long long kk = (long long)G1.nbT * k * k;
  const float sqrt_h = sqrtf((float)G1.d_out);
  if (p.lean && (ste || want_pqe || !tc || !bd_supported(BD_OUT, G1.d_out, G1.d_in, G1.ld, k, G1.g, W1) ||
                 !bd_supported(BD_IN, G2.d_out, G2.d_in, G2.ld, k, G2.g, W2))) {
    p.err = CAFEQ_ERR_WORKSPACE;  // this mode needs the matrix-sized scratch the workspace was sized without
    return;
  }
  if (tc) {
    PrepArgs pa;
    memset(&pa, 0, sizeof(pa));
    pa.M = M; pa.Mc = p.Mc; pa.Ab = p.kk.Ab; pa.kk = kk;
    pa.zero_f[0] = p.amax; pa.zero_fn[0] = 1;
    if (gradM) {
      pa.zero_f[1] = gradM; pa.zero_fn[1] = kk;
      pa.zero_f[2] = p.gMinv; pa.zero_fn[2] = kk;
    }
    pa.zero_d = p.acc; pa.zero_dn = 8;
    pa.step_counter = step_counter;
    pa.status = status;
    CQ_LAUNCH(step_prep_kernel, grid_for(kk), 256, 0, st, pa);
    if ((p.err = ns_inverse(st, p.Mc, p.Minv, G1.nbT, k, warm, p.kk, status, true, splits_kept && tb_supported(k, 2)))) return;
  } else {
    CQ_LAUNCH(zero_f64_kernel, 1, 32, 0, st, p.acc, 8);
    CQ_LAUNCH(fill_f32_kernel, 1, 32, 0, st, p.amax, 0.f, 1);
    CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, M, p.Mc, kk, status);
    if (step_counter) CQ_LAUNCH(adam_tick_kernel, 1, 1, 0, st, step_counter, status);
    launch_inverse(st, p.Mc, p.Minv, nullptr, G1.nbT, k, status);
  }
  CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, p.Minv, p.Minv_c, kk, status);
  // U = M_c^T o W1 (axis OUT), V = Minv_c o W2 (axis IN); Uhat kept in the E buffers when PQE is wanted
  const bool f1 = forward_quant(st, W1, G1, d1->bits, p.Mc, 1, p.m1, nullptr, CAFEQ_OFFSETS_NONE, false, want_pqe ? p.m1.E : nullptr, nullptr,
                nullptr, status, !force_generic);
  const bool f2 = forward_quant(st, W2, G2, d2->bits, p.Minv_c, 0, p.m2, nullptr, CAFEQ_OFFSETS_NONE, false, want_pqe ? p.m2.E : nullptr,
                nullptr, nullptr, status, !force_generic, nullptr, tc ? p.kk.Xh : nullptr, nullptr, p.tmp);  // Xh = bf16(Minv)
  const long long n1 = (long long)G1.d_out * G1.ng, n2 = (long long)G2.d_out * G2.ng;
  CQ_LAUNCH(max2_f32_kernel, grid_for(n1 + n2), 256, 0, st, p.m1.a, n1, p.m2.a, n2, p.amax, status);
  CQ_LAUNCH(sumexp2_kernel, grid_for(n1 + n2), 256, 0, st, p.m1.a, n1, p.m2.a, n2, p.amax, t, p.acc + 0, status);
  if (objective) {
    // Appendix D.1: sums of the squared group maxima; for the weighted form also ||U||_F^2 = <G1 Mc, Mc> and
    // ||V||_F^2 = <Minv_c G2, Minv_c> from the block Grams of the weights (computed once per call)
    CQ_LAUNCH(sqsum_f32_kernel, grid_for(n1), 256, 0, st, p.m1.a, n1, p.acc + 3);
    CQ_LAUNCH(sqsum_f32_kernel, grid_for(n2), 256, 0, st, p.m2.a, n2, p.acc + 4);
    if (objective == 2) {
      launch_kk(st, p.G1, 0, p.Mc, 0, p.T1, G1.nbT, k, 1.f, GEMM_STORE, status);
      launch_kk(st, p.Minv_c, 0, p.G2, 0, p.T2, G1.nbT, k, 1.f, GEMM_STORE, status);
      CQ_LAUNCH(dot_f32_kernel, grid_for(kk), 256, 0, st, p.T1, p.Mc, kk, p.acc + 5);
      CQ_LAUNCH(dot_f32_kernel, grid_for(kk), 256, 0, st, p.T2, p.Minv_c, kk, p.acc + 6);
    }
  }
  // orthonormality penalty on the fp32 parameters: R = M M^T - I (not part of the straight-through PQE loss)
  if (ste) {
  } else if (tc && p.kk.mn) {
    KkWS& w = p.kk;
    launch_split(st, M, k, kk, w.Ph, w.Pl, nullptr, nullptr, status);
    p.err = penalty_tc(st, w.Ph, w.Pl, p.RM, gradM && lambda != 0.f, p.acc + 1, 0, G1.nbT, k, status);
    if (p.err) return;
  } else if (tc) {
    // R = M M^T - I (symmetric) with its bf16 splits, ||R||_F^2, and R M for the gradient
    KkWS& w = p.kk;
    launch_split(st, M, k, kk, w.Ph, w.Pl, w.Qh, w.Ql, status);
    const uint16_t* a1[3] = {w.Ph, w.Pl, w.Ph};
    const uint16_t* b1[3] = {w.Ph, w.Ph, w.Pl};
    if ((p.err = launch_kk_tc(st, 3, a1, b1, G1.nbT, k, 1.f, 0.f, -1.f, nullptr, nullptr, w.RTh, w.RTl, nullptr, nullptr, p.acc + 1,
                 status, 0))) return;
    if (gradM && lambda != 0.f) {
      const uint16_t* a2[3] = {w.RTh, w.RTl, w.RTh};
      const uint16_t* b2[3] = {w.Qh, w.Qh, w.Ql};
      if ((p.err = launch_kk_tc(st, 3, a2, b2, G1.nbT, k, 1.f, 0.f, 0.f, nullptr, p.RM, nullptr, nullptr, nullptr, nullptr, nullptr,
                   status))) return;
    }
  } else {
    launch_kk(st, M, 0, M, 1, p.tmp, G1.nbT, k, 1.f, GEMM_STORE, status);
    CQ_LAUNCH(sub_identity_kernel, grid_for(kk), 256, 0, st, p.tmp, k, kk);
    CQ_LAUNCH(sqsum_f32_kernel, grid_for(kk), 256, 0, st, p.tmp, kk, p.acc + 1);
  }
  if (want_pqe && p.dense) {
    // Eq. 5 on the tensor cores: || Uhat_exp^T Vhat^T - P ||_F^2 with three-term bf16 splits of the dequantised values
    if ((p.err = dense_pqe(st, p.m1.E, p.m2.E, P, p.dn, p.acc + 2, nullptr, status, ste))) return;
  } else if (want_pqe) {
    launch_pair_product(st, p.m1.E, 0, G1.d_in, p.m2.E, 0, G2.d_in, G1, G2, p.R, status);
    CQ_LAUNCH(resid_sq_kernel, grid_for((long long)G1.d_in * G2.d_out), 256, 0, st, p.R, P, (long long)G1.d_in * G2.d_out, p.acc + 2,
                                                                             status);
  }
  CQ_LAUNCH(finalize_pair_kernel, 1, 1, 0, st, p.acc, p.amax, t, lambda, sqrt_h, losses, hist, ste ? 2 : (want_pqe ? 1 : 0), objective,
            (double)n1, (double)n2);
  if (!gradM) return;
  if (ste) {
    // Straight-through gradient of ||Uhat_exp^T Vhat^T - P||_F^2 (Eq. 5 squared): the residual R [d1, d3] and
    // its transpose are in p.dn.Ph/Pl/PTh/PTl; the quantiser passes gradients through except for its scale,
    // whose dependence on the group's arg-max entry is kept.
    DenseWS& w = p.dn;
    {  // g Vhat' [d3, h] = 2 R^T Uhat^T (one column for the replicas of an inner column)
      const uint16_t* a[2] = {w.PTh, w.PTl};
      const uint16_t* b[2] = {w.Awh, w.Awl};
      DenseOut o;
      o.C = w.X0T; o.ldc = w.h;
      if ((p.err = launch_dense_tc(st, 2, a, 2, b, w.d3, w.h, w.d1, 2.f, 0.f, 0.f, o, nullptr, status))) return;
    }
    {  // g Uhat [h, d1] = 2 fold(Vhat^T) R^T (the folded splits are read as they are stored: an MN-major operand costs the
      // product 10 %, 14 us, where folding, transposing and splitting again took 60)
      const uint16_t* a[2] = {w.Vh, w.Vl};
      const uint16_t* b[2] = {w.Ph, w.Pl};
      DenseOut o;
      o.C = w.U; o.ldc = w.d1;
      if ((p.err = launch_dense_tc(st, 2, a, 2, b, w.h, w.d1, w.d3, 2.f, 0.f, 0.f, o, nullptr, status, 1))) return;
    }
    if (!tc) {
      CQ_LAUNCH(fill_f32_kernel, grid_for(kk), 256, 0, st, gradM, 0.f, kk);
      CQ_LAUNCH(fill_f32_kernel, grid_for(kk), 256, 0, st, p.gMinv, 0.f, kk);
    }
    const bool og_tc = tc && ((uintptr_t)W1 % 16 == 0) && (G1.ld % 8 == 0) && ((uintptr_t)W2 % 16 == 0) && (G2.ld % 8 == 0) && G1.r == 1 &&
                       ste_split_ok(G1.g) && ste_split_ok(G2.g);
    if (og_tc) {
      // (the parts' scratch: w.U, when its splits have been taken, and w.V, which this path does not use)
      // U side (operator M^T): gradM[b][m][n] = sum_c W1[b k + m][c] gU[b k + n][c]
      launch_ste_split(st, p.m1, w.U, w.d1, G1, k, 1, qmax_of(d1->bits), w.Awh, w.Awl, status);
      if ((p.err = opgrad_out_tc(st, (const uint16_t*)W1, G1.ld, w.Awh, w.Awl, G1.nbT, k, G1.d_in, w.U, gradM, status))) return;
      // V side (operator Minv): gMinv[b][i][j] = sum over replicas and rows o of gV[o][.. + i] W2[o][.. + j]
      launch_ste_split(st, p.m2, w.X0T, w.h, G2, k, G2.r, qmax_of(d2->bits), p.gVh, p.gVl, status);
      if ((p.err = opgrad_in_tc(st, p.gVh, p.gVl, (const uint16_t*)W2, G2.ld, G1.nbT, G2.r, k, G2.d_out, w.V, p.gMinv, status))) return;
    } else {
      CQ_LAUNCH(expand_cols_kernel, dim3(w.d3, (w.h + 1023) / 1024), 256, 0, st, w.X0T, w.h, w.k, w.r, 1.f, w.V);
      const long long n1w = (long long)G1.d_out * G1.ng, n2w = (long long)G2.d_out * G2.ng;
      CQ_LAUNCH(ste_scale_path_kernel, (unsigned)((n1w * 32 + 255) / 256), 256, 0, st, p.m1.U, w.U, G1.d_in, G1.d_out, G1.ng, G1.g,
                p.m1.a, p.m1.usel, qmax_of(d1->bits), nullptr, CAFEQ_OFFSETS_NONE, G1.d_in, p.m1.coef, status);
      CQ_LAUNCH(add_argmax_kernel, grid_for(n1w), 256, 0, st, w.U, G1.d_in, G1.d_out, G1.ng, G1.g, p.m1.coef, p.m1.idx, status);
      CQ_LAUNCH(ste_scale_path_kernel, (unsigned)((n2w * 32 + 255) / 256), 256, 0, st, p.m2.U, w.V, G2.d_in, G2.d_out, G2.ng, G2.g,
                p.m2.a, p.m2.usel, qmax_of(d2->bits), nullptr, CAFEQ_OFFSETS_NONE, G2.d_in, p.m2.coef, status);
      CQ_LAUNCH(add_argmax_kernel, grid_for(n2w), 256, 0, st, w.V, G2.d_in, G2.d_out, G2.ng, G2.g, p.m2.coef, p.m2.idx, status);
      launch_opgrad(st, w.U, G1.d_in, W1, 1, G1.ld, G1, gradM, 1, 1.f, status);    // U side: operator M^T
      launch_opgrad(st, w.V, G2.d_in, W2, 1, G2.ld, G2, p.gMinv, 0, 1.f, status);  // V side: operator Minv
    }
    if (tc) {
      p.err = minv_path_tc(st, p.Minv, p.gMinv, gradM, G1.nbT, k, p.kk, status);
    } else {
      launch_kk(st, p.Minv, 1, p.gMinv, 0, p.RM, G1.nbT, k, 1.f, GEMM_STORE, status);
      launch_kk(st, p.RM, 0, p.Minv, 1, gradM, G1.nbT, k, -1.f, GEMM_STORE | GEMM_ACCUM, status);
    }
    return;
  }
  if (objective)
    CQ_LAUNCH(sumsq_coef2_kernel, grid_for(n1 + n2), 256, 0, st, p.m1.a, p.m1.usel, p.m1.coef, n1, p.m2.a, p.m2.usel, p.m2.coef, n2,
              p.acc, objective == 2 ? 1 : 0, status);
  else
    CQ_LAUNCH(lse_coef2_kernel, grid_for(n1 + n2), 256, 0, st, p.m1.a, p.m1.usel, p.m1.coef, n1, p.m2.a, p.m2.usel, p.m2.coef, n2,
              p.amax, t, p.acc + 0, status);
  if (!tc) {
    CQ_LAUNCH(fill_f32_kernel, grid_for(kk), 256, 0, st, gradM, 0.f, kk);
    CQ_LAUNCH(fill_f32_kernel, grid_for(kk), 256, 0, st, p.gMinv, 0.f, kk);
  }
  // U side: operator is M^T, so the block gradient is stored transposed
  launch_scatter(st, W1, G1, p.m1.coef, p.m1.idx, gradM, 1, status, f1 ? 1 : 0);
  // V side: gradient with respect to Minv, then through the inverse
  launch_scatter(st, W2, G2, p.m2.coef, p.m2.idx, p.gMinv, 0, status, f2 ? 1 : 0);
  if (objective == 2) {
    // mean(a_V^2) d||U||_F/dM = mean(a_V^2) G1 Mc / ||U||_F ; mean(a_U^2) d||V||_F/dMinv = mean(a_U^2) Minv_c G2 / ||V||_F
    CQ_LAUNCH(axpy_norm_kernel, grid_for(kk), 256, 0, st, gradM, p.T1, kk, p.acc, 4, (double)n2, 5, status);
    CQ_LAUNCH(axpy_norm_kernel, grid_for(kk), 256, 0, st, p.gMinv, p.T2, kk, p.acc, 3, (double)n1, 6, status);
  }
  if (tc) {
    p.err = minv_path_tc(st, p.Minv, p.gMinv, gradM, G1.nbT, k, p.kk, status);
  } else {
    launch_kk(st, p.Minv, 1, p.gMinv, 0, p.RM, G1.nbT, k, 1.f, GEMM_STORE, status);
    launch_kk(st, p.RM, 0, p.Minv, 1, gradM, G1.nbT, k, -1.f, GEMM_STORE | GEMM_ACCUM, status);
  }
  if (lambda != 0.f) {
    if (!tc) launch_kk(st, p.tmp, 0, M, 0, p.RM, G1.nbT, k, 1.f, GEMM_STORE, status);
    CQ_LAUNCH(orth_grad_kernel, grid_for(kk), 256, 0, st, gradM, p.RM, p.acc + 1, lambda, sqrt_h, kk);
  }
}

}  // namespace cafeq

#include "adaptive_offsets.cuh"

extern "C" int cafeq_workspace_size(const cafeq_matrix_desc* d1, const cafeq_matrix_desc* d2, const cafeq_opt_cfg* cfg,
                                    size_t* bytes) {
  if (!bytes) return CAFEQ_ERR_INVALID_ARG;
  if (cfg && cfg->struct_size != sizeof(cafeq_opt_cfg)) return CAFEQ_ERR_INVALID_ARG;
  Geo G1, G2;
  int rc = make_geo(d1, &G1, false);
  if (rc) return rc;
  // the sizes come from the carving code itself, run on a counting allocator
  Bump b(nullptr, 0);
  const size_t kk = (size_t)(G1.nbT > 0 ? G1.nbT : 1) * (G1.k > 0 ? G1.k : 1) * (G1.k > 0 ? G1.k : 1);
  if (!d2) {
    SingleWS s;
    carve_single(b, G1, &s, true, G1.k > 0 && lean_single_ok(G1, cfg, nullptr));
    b.take<float>(kk);  // gradient of the optimise loop / rounded operator of cafeq_rtn
  } else {
    if ((rc = make_geo(d2, &G2, false))) return rc;
    PairWS p;
    const bool lean = G1.k > 0 && G2.k > 0 && lean_pair_ok(G1, G2, cfg, nullptr, nullptr);
    carve_pair(b, G1, G2, &p, !lean, lean);
    b.take<float>(kk);
    if (!cfg) {  // cafeq_adaptive_round's learned-offset mode carves its own set of buffers from the same workspace
      Bump b2(nullptr, 0);
      LearnWS lw;
      carve_learn(b2, G1, G2, &lw);
      b2.take<float>(kk); b2.take<float>(kk); b2.take<float>(kk);
      if (b2.used > b.used) b.used = b2.used;
    }
  }
  *bytes = b.used + 256;
  return CAFEQ_OK;
}

extern "C" int cafeq_pair_product(const cafeq_matrix_desc* d1, const void* W1, const cafeq_matrix_desc* d2,
                                  const void* W2, float* P, void* ws, size_t ws_bytes, void* stream) {
  Geo G1, G2;
  int rc = make_pair_geo(d1, d2, &G1, &G2);
  if (rc) return rc;
  if (!W1 || !W2 || !P) return CAFEQ_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (ws && !((uintptr_t)ws & 255) && dense_ok(G1, G2)) {
    Bump b(ws, ws_bytes);
    DenseWS w;
    if (carve_dense(b, G1.d_out, G1.d_in, G2.d_out, G2.r, G1.k, G1.ng, G2.ng, &w)) {
      CQ_LAUNCH(bf16_to_f32_kernel, grid_for(G1.n), 256, 0, st, (const uint16_t*)W1, G1.ld, G1.d_out, G1.d_in, w.U);
      CQ_LAUNCH(bf16_to_f32_kernel, grid_for(G2.n), 256, 0, st, (const uint16_t*)W2, G2.ld, G2.d_out, G2.d_in, w.V);
      if ((rc = dense_product(st, w.U, w.V, w, P, nullptr))) return rc;
      return last_launch();
    }
  }
  launch_pair_product(st, W1, 1, G1.ld, W2, 1, G2.ld, G1, G2, P, nullptr);
  return last_launch();
}

extern "C" int cafeq_pair_loss_fwd_bwd(const cafeq_matrix_desc* d1, const void* W1, const cafeq_matrix_desc* d2,
                                       const void* W2, const float* M, const float* P, int loss_kind, float lse_t,
                                       float lambda_orth, int flags, float* losses, float* gradM, int32_t* status,
                                       void* ws, size_t ws_bytes, void* stream) {
  Geo G1, G2;
  int rc = make_pair_geo(d1, d2, &G1, &G2);
  if (rc) return rc;
  if (!W1 || !W2 || !M || !losses) return CAFEQ_ERR_INVALID_ARG;
  const bool ste = loss_kind == CAFEQ_LOSS_PQE_STE;
  const int objective = loss_kind == CAFEQ_LOSS_SUMSQ ? 1 : (loss_kind == CAFEQ_LOSS_SUMSQ_WEIGHTED ? 2 : 0);
  if (!ste && !objective && loss_kind != CAFEQ_LOSS_LSE) return CAFEQ_ERR_INVALID_ARG;
  if (ste && !dense_ok(G1, G2)) return CAFEQ_ERR_UNSUPPORTED;
  if (!(lse_t > 0.f)) return CAFEQ_ERR_INVALID_ARG;
  const bool want_grad = !(flags & CAFEQ_FLAG_NO_GRAD);
  const bool want_pqe = ste || (flags & CAFEQ_FLAG_EXACT_LOSS) != 0;
  if (want_grad && !gradM) return CAFEQ_ERR_INVALID_ARG;
  if (want_pqe && !P) return CAFEQ_ERR_INVALID_ARG;
  if ((rc = check_ws(ws, ws_bytes))) return rc;
  Bump b(ws, ws_bytes);
  PairWS p;
  if (!carve_pair(b, G1, G2, &p, want_pqe)) return CAFEQ_ERR_WORKSPACE;
  const long long kk = (long long)G1.nbT * G1.k * G1.k;
  const bool off_grad = want_grad && grad_off_16(gradM);
  float* grad = off_grad ? b.take<float>(kk) : gradM;
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  if (objective == 2) pair_grams((cudaStream_t)stream, W1, G1, W2, G2, p, status);
  pair_step((cudaStream_t)stream, d1, d2, G1, G2, W1, W2, M, P, lse_t, lambda_orth, want_pqe, losses, nullptr,
            want_grad ? grad : nullptr, status, p, (flags & CAFEQ_FLAG_GENERIC) != 0, false, nullptr, ste, objective);
  if (p.err) return p.err;
  if (off_grad) CQ_LAUNCH(copy_f32_kernel, grid_for(kk), 256, 0, (cudaStream_t)stream, grad, gradM, kk);
  return last_launch();
}

extern "C" int cafeq_optimize_pair(const cafeq_matrix_desc* d1, const void* W1, const cafeq_matrix_desc* d2,
                                   const void* W2, float* M, float* opt_state, const float* P, const cafeq_opt_cfg* cfg,
                                   float* loss_history, int32_t* status, void* ws, size_t ws_bytes, void* stream) {
  Geo G1, G2;
  int rc = make_pair_geo(d1, d2, &G1, &G2);
  if (rc) return rc;
  if (!W1 || !W2 || !M || !cfg || cfg->struct_size != sizeof(cafeq_opt_cfg) || !loss_history) return CAFEQ_ERR_INVALID_ARG;
  const bool ste = cfg->loss_kind == CAFEQ_LOSS_PQE_STE;
  const int objective = cfg->loss_kind == CAFEQ_LOSS_SUMSQ ? 1 : (cfg->loss_kind == CAFEQ_LOSS_SUMSQ_WEIGHTED ? 2 : 0);
  if ((!ste && !objective && cfg->loss_kind != CAFEQ_LOSS_LSE) || cfg->steps < 0 || !(cfg->lse_t > 0.f)) return CAFEQ_ERR_INVALID_ARG;
  if (ste && !P) return CAFEQ_ERR_INVALID_ARG;
  if (ste && !dense_ok(G1, G2)) return CAFEQ_ERR_UNSUPPORTED;
  const bool cayley = cfg->optimizer == CAFEQ_OPT_CAYLEY;
  if ((cfg->optimizer == CAFEQ_OPT_ADAM || cayley) && !opt_state) return CAFEQ_ERR_INVALID_ARG;
  if (cfg->optimizer != CAFEQ_OPT_ADAM && cfg->optimizer != CAFEQ_OPT_GD && !cayley) return CAFEQ_ERR_INVALID_ARG;
  if ((rc = check_ws(ws, ws_bytes))) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const bool any_pqe = ste || ((P != nullptr) && cfg->eval_every > 0);
  Bump b(ws, ws_bytes);
  PairWS p;
  if (!carve_pair(b, G1, G2, &p, any_pqe, !any_pqe && lean_pair_ok(G1, G2, cfg, W1, W2))) return CAFEQ_ERR_WORKSPACE;
  const long long kk = (long long)G1.nbT * G1.k * G1.k;
  float* grad = b.take<float>(kk);
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  // the inverse of the last step's transform lives in the optimiser state, so a resumed run refines it
  const bool resume = cfg->resume && opt_state;
  const StoredInverse stored(opt_state, p.Minv, kk, resume, st);
  p.Minv = stored.inv;
  if (objective == 2) pair_grams(st, W1, G1, W2, G2, p, status);
  for (int it = 0; it < cfg->steps; ++it) {
    bool eval = ste || (any_pqe && (it % cfg->eval_every == 0));
    pair_step(st, d1, d2, G1, G2, W1, W2, M, P, cfg->lse_t, cfg->lambda_orth, eval, nullptr, loss_history + 2 * (size_t)it,
              grad, status, p, false, resume || it > 0, opt_state, ste, objective, it > 0);
    if (p.err) return p.err;
    if (cayley) {
      // momentum in the state's first-moment slot
      cayley_update(st, M, grad, opt_state + CAFEQ_OPT_STATE_HEADER, cfg->lr, cfg->beta1, G1.nbT, G1.k, p, status);
    } else if (cfg->optimizer == CAFEQ_OPT_GD) {
      CQ_LAUNCH(gd_update_kernel, grid_for(kk), 256, 0, st, M, grad, cfg->lr, kk, status);
    } else {
      CQ_LAUNCH(adam_update_kernel, grid_for(kk), 256, 0, st, M, grad, opt_state, cfg->lr, cfg->beta1, cfg->beta2, cfg->eps, kk,
                                                       status);
    }
  }
  stored.keep(cfg->steps);
  return last_launch();
}

extern "C" int cafeq_adaptive_round(const cafeq_matrix_desc* d1, const void* W1, const cafeq_matrix_desc* d2,
                                    const void* W2, const float* M, int iters, int mode, int8_t* codes1, float* scales1,
                                    int8_t* codes2, float* scales2, float* pqe_history, int32_t* status, void* ws,
                                    size_t ws_bytes, void* stream) {
  Geo G1, G2;
  int rc = make_pair_geo(d1, d2, &G1, &G2);
  if (rc) return rc;
  if (!W1 || !W2 || !codes1 || !scales1 || !codes2 || !scales2 || !pqe_history) return CAFEQ_ERR_INVALID_ARG;
  if (mode != CAFEQ_ROUND_ALG1 && mode != CAFEQ_ROUND_LEARNED_OFFSETS) return CAFEQ_ERR_INVALID_ARG;
  if (iters < 0 || iters > (mode == CAFEQ_ROUND_ALG1 ? 15 : 30)) return CAFEQ_ERR_INVALID_ARG;
  if ((rc = check_ws(ws, ws_bytes))) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (mode == CAFEQ_ROUND_LEARNED_OFFSETS) {
    if (iters < 1) return CAFEQ_ERR_INVALID_ARG;
    Bump b(ws, ws_bytes);
    LearnWS w;
    carve_learn(b, G1, G2, &w);
    const long long kk = (long long)G1.nbT * G1.k * G1.k;
    float* Mc = b.take<float>(kk);
    float* Minv = b.take<float>(kk);
    float* Minv_c = b.take<float>(kk);
    if (b.overflow) return CAFEQ_ERR_WORKSPACE;
    if (M) {
      CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, M, Mc, kk, status);
      launch_inverse(st, Mc, Minv, nullptr, G1.nbT, G1.k, status);
      CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, Minv, Minv_c, kk, status);
      launch_apply(st, W1, 1, G1.ld, G1, Mc, 1, w.U, G1.d_in, GEMM_STORE, nullptr, status);
      launch_apply(st, W2, 1, G2.ld, G2, Minv_c, 0, w.V, G2.d_in, GEMM_STORE, nullptr, status);
    } else {
      CQ_LAUNCH(bf16_to_f32_kernel, grid_for(G1.n), 256, 0, st, (const uint16_t*)W1, G1.ld, G1.d_out, G1.d_in, w.U);
      CQ_LAUNCH(bf16_to_f32_kernel, grid_for(G2.n), 256, 0, st, (const uint16_t*)W2, G2.ld, G2.d_out, G2.d_in, w.V);
    }
    learned_offsets_run(st, d1->bits, G1, G2, iters, codes1, scales1, codes2, scales2, pqe_history, w, status);
    return last_launch();
  }
  if (!dense_ok(G1, G2)) return CAFEQ_ERR_UNSUPPORTED;  // every dimension a multiple of 64, block a multiple of 32
  Bump b(ws, ws_bytes);
  DenseWS w;
  if (!carve_dense(b, G1.d_out, G1.d_in, G2.d_out, G2.r, G1.k, G1.ng, G2.ng, &w)) return CAFEQ_ERR_WORKSPACE;
  const long long kk = (long long)G1.nbT * G1.k * G1.k;
  float* Mc = b.take<float>(kk);
  float* Minv = b.take<float>(kk);
  float* Minv_c = b.take<float>(kk);
  KkWS kkw;
  carve_kk(b, G1.nbT, G1.k, &kkw);
  if (b.overflow) return CAFEQ_ERR_WORKSPACE;
  if (M) {
    // the transformed pair U = W1 M (operator bf16(M)^T on the stored rows), V = M^-1 W2 (operator bf16(inv(bf16(M))))
    CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, M, Mc, kk, status);
    // block sizes 128 / 256: elimination takes 5 ms at k = 256 (one CTA per block, k dependent steps); at k <= 64 it is
    // short and stays
    if (tb_supported(G1.k, 2)) {
      if ((rc = ns_inverse(st, Mc, Minv, G1.nbT, G1.k, false, kkw, status))) return rc;
    } else launch_inverse(st, Mc, Minv, nullptr, G1.nbT, G1.k, status);
    CQ_LAUNCH(round_bf16_kernel, grid_for(kk), 256, 0, st, Minv, Minv_c, kk, status);
    // both products on the tensor cores where the shape allows (bf16 operands, fp32 accumulation either way); the operators in
    // applied orientation use scratch that nothing else needs here
    uint16_t *T1 = kkw.Ph, *T2 = kkw.Qh;
    launch_operator_bf16(st, Mc, T1, G1.k, G1.nbT, 1, status);
    launch_operator_bf16(st, Minv_c, T2, G1.k, G1.nbT, 0, status);
    if (!apply_tc(st, W1, G1, T1, w.U, status)) launch_apply(st, W1, 1, G1.ld, G1, Mc, 1, w.U, G1.d_in, GEMM_STORE, nullptr, status);
    if (!apply_tc(st, W2, G2, T2, w.V, status)) launch_apply(st, W2, 1, G2.ld, G2, Minv_c, 0, w.V, G2.d_in, GEMM_STORE, nullptr, status);
  } else {
    CQ_LAUNCH(bf16_to_f32_kernel, grid_for(G1.n), 256, 0, st, (const uint16_t*)W1, G1.ld, G1.d_out, G1.d_in, w.U);
    CQ_LAUNCH(bf16_to_f32_kernel, grid_for(G2.n), 256, 0, st, (const uint16_t*)W2, G2.ld, G2.d_out, G2.d_in, w.V);
  }
  if ((rc = alg1_run(st, d1->bits, G1.g, G2.g, iters, codes1, scales1, codes2, scales2, pqe_history, w, status))) return rc;
  return last_launch();
}

extern "C" int cafeq_pack(const cafeq_matrix_desc* d, const int8_t* codes, uint8_t* packed, void* stream) {
  Geo G;
  int rc = make_geo(d, &G, false);
  if (rc) return rc;
  if (!codes || !packed) return CAFEQ_ERR_INVALID_ARG;
  if (G.d_in % 8) return CAFEQ_ERR_UNSUPPORTED;
  if (G.d_in % 32 == 0 && ((uintptr_t)codes % 16) == 0 && ((uintptr_t)packed % 4) == 0 && d->bits >= 2 && d->bits <= 8) {
    cudaStream_t ps = (cudaStream_t)stream;
    const unsigned pg = grid_for(G.n / 32);
    uint32_t* pw = reinterpret_cast<uint32_t*>(packed);
    switch (d->bits) {
      case 2: CQ_LAUNCH(pack32_kernel<2>, pg, 256, 0, ps, codes, pw, G.d_out, G.d_in); break;
      case 3: CQ_LAUNCH(pack32_kernel<3>, pg, 256, 0, ps, codes, pw, G.d_out, G.d_in); break;
      case 4: CQ_LAUNCH(pack32_kernel<4>, pg, 256, 0, ps, codes, pw, G.d_out, G.d_in); break;
      case 5: CQ_LAUNCH(pack32_kernel<5>, pg, 256, 0, ps, codes, pw, G.d_out, G.d_in); break;
      case 6: CQ_LAUNCH(pack32_kernel<6>, pg, 256, 0, ps, codes, pw, G.d_out, G.d_in); break;
      case 7: CQ_LAUNCH(pack32_kernel<7>, pg, 256, 0, ps, codes, pw, G.d_out, G.d_in); break;
      default: CQ_LAUNCH(pack32_kernel<8>, pg, 256, 0, ps, codes, pw, G.d_out, G.d_in); break;
    }
    return last_launch();
  }
  CQ_LAUNCH(pack_kernel, grid_for(G.n / 8), 256, 0, (cudaStream_t)stream, codes, packed, G.d_out, G.d_in, d->bits);
  return last_launch();
}

#include "layer_step.cuh"

// ------------------------------------------------------------------------------------------------
// cafeq_rtn without a caller workspace: scratch lives in the library image
// ------------------------------------------------------------------------------------------------
// In host code the name of a __device__ array is only a handle for the runtime, not an address a kernel can
// use; the device address is looked up once per device with cudaGetSymbolAddress and cached.
static __device__ __align__(256) unsigned char g_noalloc_scratch[CAFEQ_NOALLOC_SCRATCH_BYTES];
static constexpr int kMaxDevices = 64;
static void* g_noalloc_ptr[kMaxDevices] = {};
static std::mutex g_noalloc_mu;

extern "C" int cafeq_rtn_noalloc(const cafeq_matrix_desc* d, const void* W, const float* T, int8_t* codes, float* scales,
                                 void* stream) {
  Geo Gq;
  int rc = make_geo(d, &Gq, false);
  if (rc) return rc;
  if (!W || !codes || !scales) return CAFEQ_ERR_INVALID_ARG;
  // what cafeq_rtn would carve for this very call (cafeq_rtn_workspace_size gives the same figure for aligned buffers)
  const size_t need = rtn_scratch(Gq, T != nullptr && Gq.k > 0, W, codes, nullptr, nullptr, nullptr);
  if (need > (size_t)CAFEQ_NOALLOC_SCRATCH_BYTES) return CAFEQ_ERR_TOO_LARGE;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return CAFEQ_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return CAFEQ_ERR_UNSUPPORTED;
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return CAFEQ_ERR_CUDA;
      g_noalloc_ptr[dev] = p;
    }
    scratch = g_noalloc_ptr[dev];
  }
  return cafeq_rtn(d, W, T, codes, scales, scratch, (size_t)CAFEQ_NOALLOC_SCRATCH_BYTES, stream);
}
