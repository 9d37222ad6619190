// Host side of the dense pair algebra: the product term of Eq. 5 (PQE) and Algorithm 1 (adaptive rounding),
// built from the tensor-core product kernel with three-term bf16 splits (fp32-grade accuracy).
// Included by cafeq_api.cu (uses its launch counter, workspace carving and quantiser launch helpers).
#pragma once

#include "kernels_dense.cuh"
#include "kernels_gemm2.cuh"

namespace cafeq {

// C = alpha * sum_t A_t B_t^T + beta * C0 + gamma * I  for one dense product (no batching)
struct DenseOut {
  const float* C0 = nullptr;
  long long ldc0 = 0;
  float* C = nullptr;
  long long ldc = 0;
  uint16_t *Chi = nullptr, *Clo = nullptr, *Cthi = nullptr, *Ctlo = nullptr;
  double* sq = nullptr;
  const double* stop_sq = nullptr;  // stopping rule of an iteration (TgParams)
  int stop_it = 0, stop_guard = 0;
};

static TgParams dense_params(int M, int N, int K, float alpha, float beta, float gamma, const DenseOut& o, int32_t* status, int a_mn) {
  TgParams p;
  memset(&p, 0, sizeof(p));
  p.M = M; p.N = N; p.K = K;
  p.batch = 1;
  p.divA = 1;
  p.alpha = alpha; p.beta = beta; p.gamma = gamma;
  p.C0 = o.C0; p.ldc0 = o.ldc0;
  p.C = o.C; p.ldc = o.ldc;
  p.Chi = o.Chi; p.Clo = o.Clo; p.Cthi = o.Cthi; p.Ctlo = o.Ctlo;
  p.sq = o.sq; p.sq_stride = 0;
  p.a_mn = a_mn;
  p.stop_sq = o.stop_sq; p.stop_it = o.stop_it; p.stop_guard = o.stop_guard;
  p.status = status;
  return p;
}

// One launch of up to three terms on the tiled kernel, in the order given.
static int tg_launch_dense(cudaStream_t st, int nterms, const uint16_t* const* A, const uint16_t* const* B, int M, int N, int K,
                              float alpha, float beta, float gamma, const DenseOut& o, int32_t* status, int a_mn) {
  TgOperand oa[TG_MAX_TERMS], ob[TG_MAX_TERMS];
  for (int t = 0; t < nterms; ++t) {
    oa[t] = a_mn ? TgOperand{A[t], K, M, M} : TgOperand{A[t], M, K, K};
    ob[t] = TgOperand{B[t], N, K, K};
  }
  TgParams p = dense_params(M, N, K, alpha, beta, gamma, o, status, a_mn);
  p.nterms = nterms;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return tg_launch(st, oa, ob, p);
}

// C = alpha * A B^T + beta * C0 + gamma * I with A [M, K] (a_mn: [K, M]) and B [N, K] given as sums of na and nb bf16 arrays
// ({hi, lo}: 16 significand bits, {hi, lo, third}: 24): the terms A_i B_j with i + j < max(na, nb).  With two arrays each these
// are three terms (fp32-grade to about 2^-17 per entry), with three each six, down to 2^-24: what is left is the rounding of the
// fp32 accumulators.  acc: fp32 [M, N] for the first half of more than three terms on the tiled kernel (it may be o.C).
//
// Six terms, and three with a long contraction, run on CTA pairs (t2_wanted).
static int launch_dense_tc(cudaStream_t st, int na, const uint16_t* const* A, int nb, const uint16_t* const* B, int M, int N, int K,
                        float alpha, float beta, float gamma, const DenseOut& o, float* acc, int32_t* status, int a_mn = 0) {
  const int order = na > nb ? na : nb;
  double cost;
  const int bn = t2_width(M, N, 0, &cost);
  if (K % TG_BK == 0 && t2_wanted(M, N, K, order, cost)) {
    T2Maps maps;
    T2Params tp;
    memset(&maps, 0, sizeof(maps));
    memset(&tp, 0, sizeof(tp));
    bool ok = true;
    for (int i = 0; i < na; ++i)
      ok = ok && make_map_bf16(&maps.a[0][i], A[i], a_mn ? M : K, a_mn ? K : M, a_mn ? M : K, a_mn ? 64 : 128);
    for (int j = 0; j < nb; ++j) ok = ok && make_map_bf16(&maps.b[j], B[j], K, N, K, bn / 2);
    if (ok) {
      tp.p[0] = dense_params(M, N, K, alpha, beta, gamma, o, status, a_mn);
      tp.nprob = 1;
      tp.sh = t2_shape(M, N, bn, na, nb, order);
      g_launches.fetch_add(1, std::memory_order_relaxed);
      return t2_launch(st, maps, tp);
    }
  }
  // The small terms first: every addition to an accumulator is rounded at the accumulator's size, so small terms that follow the
  // large ones cost as much accuracy as those.  Product of bf16 weights with two replicas folded (their sums have a second term),
  // 2048 x 3584 x 3584, against float64: 2.0e-6, large terms first 6.0e-6.
  const uint16_t* a1[3] = {A[1], A[0], A[0]};
  const uint16_t* b1[3] = {B[0], B[1], B[0]};
  if (order == 2) return tg_launch_dense(st, 3, a1, b1, M, N, K, alpha, beta, gamma, o, status, a_mn);
  DenseOut o1;
  o1.C0 = o.C0; o1.ldc0 = o.ldc0;
  o1.C = acc; o1.ldc = N;
  int rc = tg_launch_dense(st, 3, a1, b1, M, N, K, alpha, beta, gamma, o1, status, a_mn);
  if (rc) return rc;
  const uint16_t* a2[3];
  const uint16_t* b2[3];
  int n2 = 0;
  if (nb > 2) { a2[n2] = A[0]; b2[n2++] = B[2]; }
  if (na > 2) { a2[n2] = A[2]; b2[n2++] = B[0]; }
  a2[n2] = A[1]; b2[n2++] = B[1];
  DenseOut o2 = o;
  o2.C0 = acc; o2.ldc0 = N;
  return tg_launch_dense(st, n2, a2, b2, M, N, K, alpha, 1.f, 0.f, o2, status, a_mn);
}

static void launch_split_rect(cudaStream_t st, const float* X, int R, int C, long long ld, float scale, const double* inv_scale,
                              float* Y, float* YT, uint16_t* hi, uint16_t* lo, uint16_t* thi, uint16_t* tlo, const int32_t* status,
                              uint16_t* h3 = nullptr, uint16_t* t3 = nullptr, const double* norm2 = nullptr) {
  CQ_LAUNCH(split_rect_kernel, dim3(C / 64, R / 64), 256, 0, st, X, R, C, ld, scale, inv_scale, Y, YT, hi, lo, thi, tlo, status, h3, t3, norm2);
}

// Scratch of the dense pair algebra for a pair with stored shapes U [h, d1], V [d3, rh]
struct DenseWS {
  int h, d1, d3, rh, k, r, D;
  float *U, *V, *Uhat, *Vhat, *P, *Bf, *X0T, *Y;
  uint16_t *Ph, *Pl, *PTh, *PTl;          // P [d1, d3] and its transpose [d3, d1]
  uint16_t *UTh, *UTl;                    // transposed splits of a [h, d1] matrix: [d1, h]
  uint16_t *Vh, *Vl;                      // splits of a [d3, rh] matrix
  uint16_t *Awh, *Awl;                    // the (wide) matrix being pseudo-inverted [m, n]
  uint16_t *Yh, *Yl, *YTh[2], *YTl[2];    // iterate Y = X^T [m, n] and its transpose [n, m]
  uint16_t *CTh, *CTl;                    // transposed residual [m, m]
  uint16_t *Oh, *Ol, *O3;                 // pseudo-inverse result in the stored shape [h, D], split three ways
  uint16_t *P3, *PT3, *UT3, *V3, *Aw3, *Y3;  // third terms of the operands that take part in six-term products
  float* Cf;                              // fp32 accumulator of a six-term product [max(m, d1, d3), ...]
  float *qa, *qusel;                      // quantiser scratch: absmax, signed arg-max value
  int* qidx;
  double* sq;                             // [DENSE_SQ] accumulators: 0..: PQE history, 32..: iteration residuals
};
constexpr int DENSE_SQ = 128;
constexpr int PINV_MAX_ITERS = 60;

static bool carve_dense(Bump& b, int h, int d1, int d3, int r, int k, int ng1, int ng2, DenseWS* w) {
  const size_t rh = (size_t)r * h, D = (size_t)(d1 > d3 ? d1 : d3);
  w->h = h; w->d1 = d1; w->d3 = d3; w->rh = (int)rh; w->k = k; w->r = r; w->D = (int)D;
  const size_t nU = (size_t)h * d1, nV = (size_t)d3 * rh, nP = (size_t)d1 * d3, nY = (size_t)h * D;
  const size_t m = (size_t)h < D ? (size_t)h : D;  // smaller side of any matrix that gets pseudo-inverted
  w->U = b.take<float>(nU); w->V = b.take<float>(nV);
  w->Uhat = b.take<float>(nU); w->Vhat = b.take<float>(nV);
  w->P = b.take<float>(nP);
  w->Bf = b.take<float>((size_t)h * d3);
  w->X0T = b.take<float>((size_t)d3 * h);
  w->Y = b.take<float>(nY);
  w->Ph = b.take<uint16_t>(nP); w->Pl = b.take<uint16_t>(nP); w->PTh = b.take<uint16_t>(nP); w->PTl = b.take<uint16_t>(nP);
  w->UTh = b.take<uint16_t>(nU); w->UTl = b.take<uint16_t>(nU);
  w->Vh = b.take<uint16_t>(nV); w->Vl = b.take<uint16_t>(nV);
  w->Awh = b.take<uint16_t>(nY); w->Awl = b.take<uint16_t>(nY);
  w->Yh = b.take<uint16_t>(nY); w->Yl = b.take<uint16_t>(nY);
  for (int q = 0; q < 2; ++q) { w->YTh[q] = b.take<uint16_t>(nY); w->YTl[q] = b.take<uint16_t>(nY); }
  w->CTh = b.take<uint16_t>(m * m); w->CTl = b.take<uint16_t>(m * m);
  w->Oh = b.take<uint16_t>(nY); w->Ol = b.take<uint16_t>(nY); w->O3 = b.take<uint16_t>(nY);
  w->P3 = b.take<uint16_t>(nP); w->PT3 = b.take<uint16_t>(nP);
  w->UT3 = b.take<uint16_t>(nU); w->V3 = b.take<uint16_t>(nV);
  w->Aw3 = b.take<uint16_t>(nY); w->Y3 = b.take<uint16_t>(nY);
  w->Cf = b.take<float>(m * m > nY ? m * m : nY);
  const size_t nq = ((size_t)h * ng1 > (size_t)d3 * ng2) ? (size_t)h * ng1 : (size_t)d3 * ng2;
  w->qa = b.take<float>(nq); w->qusel = b.take<float>(nq); w->qidx = b.take<int>(nq);
  w->sq = b.take<double>(DENSE_SQ);
  return !b.overflow;
}

// Approximate G^-1 = (A A^T)^-1 for the splits of A in w.Aw* ([m, n], m <= n), left as bf16 splits in w.CTh / w.CTl.
// Y <- 2 mu Y - mu^2 Y B and B <- 2 mu B - mu^2 B B from B = G / c (c a little above ||G||_F), Y = I / c: B = G Y c throughout, and
// with mu = 2 / (1 + l) for the smallest eigenvalue l of B the eigenvalues of B go to 1, l growing fourfold a step at first.
// Both are polynomials in G, so one launch does both products on their upper tiles: 36 + 36 pairs at m = 2048, one wave, 45 us; a
// step of the rectangular iteration takes 160.  l starts at 2^-13: smaller eigenvalues grow as far as that and are finished by the
// rectangular iteration (the products' errors grow with them, fourfold a step: from 2^-14 they left residuals twice as large).
// Nothing here need be accurate: whatever Y is, A^T Y lies in the row space of A, and its error is what the rectangular iteration
// corrects.
// The Y of gram_restart(m) steps is kept in w.Oh / w.Ol for the restart (pinv_rows); the steps after it are skipped on a matrix with a
// row of zeros.
constexpr int GRAM_STEPS = 9;
static int gram_restart(int m) { return m < 512 ? 1 : 2; }
static int gram_inverse(cudaStream_t st, int m, int n, DenseWS& w, double* fro2, double* rs, double* singular, int32_t* status) {
  T2Maps maps;
  T2Params tp;
  int rc;
  const uint16_t* aw[2] = {w.Awh, w.Awl};
  memset(&maps, 0, sizeof(maps));
  memset(&tp, 0, sizeof(tp));
  for (int i = 0; i < 2; ++i)
    if (!make_map_bf16(&maps.a[0][i], aw[i], n, m, n, 128) || !make_map_bf16(&maps.b[i], aw[i], n, m, n, 128)) return CAFEQ_ERR_UNSUPPORTED;
  DenseOut g;
  g.C = w.Y; g.ldc = m; g.sq = fro2;
  tp.p[0] = dense_params(m, m, n, 1.f, 0.f, 0.f, g, status, 0);
  tp.nprob = 1;
  tp.sh = t2_shape(m, m, 256, 2, 2, 2);
  tp.sh.sym = 1;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if ((rc = t2_launch(st, maps, tp))) return rc;
  uint16_t* Bs[2][2] = {{w.Yh, w.Yl}, {w.YTh[0], w.YTl[0]}};
  uint16_t* Ys[2][2] = {{w.YTh[1], w.YTl[1]}, {w.CTh, w.CTl}};
  uint16_t* kept[2] = {w.Oh, w.Ol};
  const int keep = gram_restart(m);
  static_assert(GRAM_STEPS % 2 == 1, "the result is left in the second pair of buffers");
  double l = 1.0 / 8192.0;
  for (int j = 0; j < GRAM_STEPS; ++j) {
    const float mu = (float)(2.0 / (1.0 + l));
    l = 4.0 * l / ((1.0 + l) * (1.0 + l));
    if (j == 0)
      CQ_LAUNCH(gram_start_kernel, dim3(m / 64, m / 64), 256, 0, st, w.Y, m, fro2, mu, w.Cf, Bs[0][0], Bs[0][1],
                keep == 1 ? kept[0] : Ys[1][0], keep == 1 ? kept[1] : Ys[1][1], singular, rs, status);
    const int b = j & 1;
    tp.nprob = 0;
    auto add = [&](uint16_t* const* from, uint16_t* const* to, float* X) {
      DenseOut o;
      o.C0 = X; o.ldc0 = m; o.C = X; o.ldc = m;
      o.Chi = to[0]; o.Clo = to[1];
      if (j >= keep) { o.stop_sq = singular; o.stop_guard = 16; }
      tp.p[tp.nprob] = dense_params(m, m, m, -mu * mu, 2.f * mu, 0.f, o, status, 0);
      for (int i = 0; i < 2; ++i)
        if (!make_map_bf16(&maps.a[tp.nprob][i], from[i], m, m, m, 128)) return false;
      ++tp.nprob;
      return true;
    };
    if (j + 1 < GRAM_STEPS && !add(Bs[b], Bs[b ^ 1], w.Y)) return CAFEQ_ERR_UNSUPPORTED;
    if (j > 0 && !add(j == keep ? kept : Ys[b], j + 1 == keep ? kept : Ys[b ^ 1], w.Cf)) return CAFEQ_ERR_UNSUPPORTED;
    for (int i = 0; i < 2; ++i)
      if (!make_map_bf16(&maps.b[i], Bs[b][i], m, m, m, 128)) return CAFEQ_ERR_UNSUPPORTED;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if ((rc = t2_launch(st, maps, tp))) return rc;
  }
  return CAFEQ_OK;
}

// out (hi / lo, shape [R, C] of S) = pinv(S^T) = pinv(S)^T on the wide orientation A of S ([m, n], m <= n), carried as Y = X^T so
// that every product has both operands contraction-major.  A is S times a power of two that brings its norm to [1, 2): the norm of
// its Gram matrix is taken from sums of fourth powers, which leave the range of fp32 at row norms of 4e9 and 1e-11.  The same power
// brings the result back.
//   1. X0 = A^T G^-1 with the approximate inverse of the Gram matrix (gram_inverse), as five terms over A split three ways: the
//      iteration below never corrects what lies outside the row space of A, so X0 must not leave it.
//   2. Newton-Schulz X <- X + X (I - A X), until an update that began below ||I - A X||_F = 1e-3 or until one would begin below
//      2^-12 (step 3 squares it), or until the residual stalls, which every product works out from the residuals itself.  One or two
//      updates for the 9B-shaped v-o factors (kappa^2 some thousands) instead of the sixteen from X0 = A^T / c.
//   3. One step with the residual over three-way splits.
// When A X0 is not within 0.9 of I (rank-deficient or very badly conditioned A) the iteration restarts from X0 = A^T Y with the Y of
// one or two Gram steps: the eigenvalues of A X0 lie in [0, 1], and it converges to the Moore-Penrose inverse (stalling at the rank
// defect).  Each Gram step saves two iterations, and lets Y grow fourfold where A A^T is singular; there A^T Y cancels only to the
// rounding of what cancels.  With 4^steps about the square root of m that stays below the rounding of the iteration itself: against
// float64, 64 x 192 with one of its rows repeated, scales off by 1.4e-7 after one step (none 2.3e-7), 3.1e-6 after four.
// Error against a float64 pseudo-inverse (512 x 768, kappa^2 4000, emulated products): 1.3e-7; from X0 = A^T / c 7e-6.
static int pinv_rows(cudaStream_t st, const float* S, int R, int C, DenseWS& w, int32_t* status) {
  const bool wide = R <= C;
  const int m = wide ? R : C, n = wide ? C : R;
  double* fro2 = w.sq + 120;
  double* norm2 = w.sq + 121;
  double* singular = w.sq + 122;
  double* rs = w.sq + 32;  // residuals per iteration
  int rc;
  CQ_LAUNCH(zero_f64_kernel, 1, 128, 0, st, w.sq + 32, DENSE_SQ - 32);
  CQ_LAUNCH(sqsum_f32_kernel, grid_for((long long)R * C), 256, 0, st, S, (long long)R * C, norm2);
  if (wide) launch_split_rect(st, S, R, C, C, 1.f, nullptr, nullptr, nullptr, w.Awh, w.Awl, nullptr, nullptr, status, w.Aw3, nullptr, norm2);
  else launch_split_rect(st, S, R, C, C, 1.f, nullptr, nullptr, nullptr, nullptr, nullptr, w.Awh, w.Awl, status, nullptr, w.Aw3, norm2);
  if ((rc = gram_inverse(st, m, n, w, fro2, rs, singular, status))) return rc;
  // Y = (g0 + g1) A (the rows of A, the contraction, are read as they are stored)
  auto start = [&](const uint16_t* g0, const uint16_t* g1, int cur, const double* sq, int guard) -> int {
    const uint16_t* g[2] = {g0, g1};
    const uint16_t* a[3] = {w.Awh, w.Awl, w.Aw3};
    const int bn = t2_width(m, n, 1, nullptr);
    T2Maps maps;
    T2Params tp;
    memset(&maps, 0, sizeof(maps));
    memset(&tp, 0, sizeof(tp));
    bool ok = true;
    for (int i = 0; i < 2; ++i) ok = ok && make_map_bf16(&maps.a[0][i], g[i], m, m, m, 128);
    for (int i = 0; i < 3; ++i) ok = ok && make_map_bf16(&maps.b[i], a[i], n, m, n, 64);
    if (!ok) return CAFEQ_ERR_UNSUPPORTED;
    DenseOut o;
    o.C = w.Y; o.ldc = n;
    o.Chi = w.Yh; o.Clo = w.Yl; o.Cthi = w.YTh[cur]; o.Ctlo = w.YTl[cur];
    o.stop_sq = sq; o.stop_guard = guard;
    tp.p[0] = dense_params(m, n, m, 1.f, 0.f, 0.f, o, status, 0);
    tp.p[0].b_mn = 1;
    tp.nprob = 1;
    tp.sh = t2_shape(m, n, bn, 2, 3, 3);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return t2_launch(st, maps, tp);
  };
  if ((rc = start(w.CTh, w.CTl, 0, singular, 16))) return rc;
  const uint16_t* aw[2] = {w.Awh, w.Awl};
  const uint16_t* ct[2] = {w.CTh, w.CTl};
  const uint16_t* y[2] = {w.Yh, w.Yl};
  auto residual = [&](DenseOut& o) { o.Cthi = w.CTh; o.Ctlo = w.CTl; o.sq = rs; o.stop_sq = rs; o.stop_guard = 1; };  // C = I - A X, kept transposed
  auto update = [&](DenseOut& o, int cur) {                                                      // Y += C^T Y
    o.C0 = w.Y; o.ldc0 = n; o.C = w.Y; o.ldc = n;
    o.Chi = w.Yh; o.Clo = w.Yl; o.Cthi = w.YTh[cur ^ 1]; o.Ctlo = w.YTl[cur ^ 1];
    o.stop_sq = rs; o.stop_guard = 5;
  };
  constexpr int LAUNCHED = 3;
  for (int it = 0; it < LAUNCHED; ++it) {
    const int cur = it & 1;
    DenseOut o;
    residual(o);
    o.sq = rs + it; o.stop_it = it;
    if ((rc = launch_dense_tc(st, 2, aw, 2, y, m, m, n, -1.f, 0.f, 1.f, o, nullptr, status))) return rc;
    const uint16_t* yt[2] = {w.YTh[cur], w.YTl[cur]};
    DenseOut u;
    update(u, cur);
    u.stop_it = it;
    if (it == 0) u.stop_guard = 7;
    if ((rc = launch_dense_tc(st, 2, ct, 2, yt, m, n, m, 1.f, 1.f, 0.f, u, nullptr, status))) return rc;
    if (it == 0 && (rc = start(w.Oh, w.Ol, 1, rs, 8))) return rc;  // the restart: what update 0 would have written
  }
  {
    T2LoopMaps maps;
    T2LoopParams lp;
    memset(&maps, 0, sizeof(maps));
    memset(&lp, 0, sizeof(lp));
    // (narrow tiles where there are few: with these and without the barriers that the grid's include an iteration of 256 x 512 takes 18
    // us, of tiles of 128 columns and more 25)
    const int bm = t2_width(m, m, 0, nullptr, 64), bn = t2_width(m, n, 0, nullptr, 64);
    bool ok = true;
    for (int i = 0; i < 2; ++i) {
      ok = ok && make_map_bf16(&maps.a[0][i], aw[i], n, m, n, 128) && make_map_bf16(&maps.b[0][i], y[i], n, m, n, bm / 2);
      ok = ok && make_map_bf16(&maps.a[1][i], ct[i], m, m, m, 128);
      for (int cur = 0; cur < 2; ++cur) ok = ok && make_map_bf16(&maps.b[1 + cur][i], i ? w.YTl[cur] : w.YTh[cur], m, n, m, bn / 2);
    }
    if (!ok) return CAFEQ_ERR_UNSUPPORTED;
    for (int cur = 0; cur < 2; ++cur) {
      DenseOut o, u;
      residual(o);
      update(u, cur);
      lp.p[0][cur] = dense_params(m, m, n, -1.f, 0.f, 1.f, o, status, 0);
      lp.p[1][cur] = dense_params(m, n, m, 1.f, 1.f, 0.f, u, status, 0);
    }
    lp.sh[0] = t2_shape(m, m, bm, 2, 2, 2);
    lp.sh[1] = t2_shape(m, n, bn, 2, 2, 2);
    lp.it0 = LAUNCHED; lp.it1 = PINV_MAX_ITERS;
    lp.arrived = reinterpret_cast<uint32_t*>(w.sq + 124);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if ((rc = pinv_loop_launch(st, maps, lp))) return rc;
  }
  // The loop above stops at a residual of 2^-12 at most (Frobenius), in the accuracy of its three-term products.  One more
  // step with the residual evaluated over three-way splits (fp32-grade) squares what is left: the quantised targets
  // of Algorithm 1 then agree with a float64 pseudo-inverse except at rounding ties.  The correction C^T Y is small,
  // three terms are enough for it.  (A rank-deficient matrix stalls where it stalled before: the step changes nothing.)
  {
    launch_split_rect(st, w.Y, m, n, n, 1.f, nullptr, nullptr, nullptr, w.Yh, w.Yl, w.YTh[0], w.YTl[0], status, w.Y3, nullptr);
    const uint16_t* a[3] = {w.Awh, w.Awl, w.Aw3};
    const uint16_t* bb[3] = {w.Yh, w.Yl, w.Y3};
    DenseOut o;
    o.Cthi = w.CTh; o.Ctlo = w.CTl;
    if ((rc = launch_dense_tc(st, 3, a, 3, bb, m, m, n, -1.f, 0.f, 1.f, o, w.Cf, status))) return rc;
    const uint16_t* a2[2] = {w.CTh, w.CTl};
    const uint16_t* b2[2] = {w.YTh[0], w.YTl[0]};
    DenseOut o2;
    o2.C0 = w.Y; o2.ldc0 = n; o2.C = w.Y; o2.ldc = n;
    if ((rc = launch_dense_tc(st, 2, a2, 2, b2, m, n, m, 1.f, 1.f, 0.f, o2, nullptr, status))) return rc;
  }
  if (wide) launch_split_rect(st, w.Y, m, n, n, 1.f, nullptr, nullptr, nullptr, w.Oh, w.Ol, nullptr, nullptr, status, w.O3, nullptr, norm2);
  else launch_split_rect(st, w.Y, m, n, n, 1.f, nullptr, nullptr, nullptr, nullptr, nullptr, w.Oh, w.Ol, status, nullptr, w.O3, norm2);
  return CAFEQ_OK;
}

}  // namespace cafeq

namespace cafeq {

// Group quantiser on an fp32 matrix T [rows, cols] (groups of g along the row): codes, scales, dequantised values
static void quant_matrix(cudaStream_t st, const float* T, int rows, int cols, int g, int bits, int8_t* codes, float* scales,
                         float* That, DenseWS& w, int32_t* status) {
  launch_group_quant(st, T, cols, rows, cols / g, g, qmax_of(bits), nullptr, CAFEQ_OFFSETS_NONE, w.qa, w.qusel, w.qidx, nullptr, That,
                     codes, scales, status);
}

// hi / lo (and third) terms of V [d3, rh] with its replicas folded: [d3, h]
static void launch_fold_split(cudaStream_t st, const float* V, DenseWS& w, uint16_t* hi, uint16_t* lo, uint16_t* h3, int32_t* status) {
  CQ_LAUNCH(fold_split_kernel, dim3(w.d3, (w.h + 1023) / 1024), 256, 0, st, V, w.h, w.k, w.r, hi, lo, h3, status);
}

// P = U_exp^T V^T for stored U [h, d1], V [d3, rh] (fp32): fp32 P [d1, d3] with its splits in w.Ph/Pl/PTh/PTl
// (six terms over three-way splits: P is the reference every least-squares target of Algorithm 1 is measured
// against, so it is formed to fp32 accuracy; its own third-term splits follow for the target products)
static int dense_product(cudaStream_t st, const float* U, const float* V, DenseWS& w, float* P, int32_t* status) {
  launch_split_rect(st, U, w.h, w.d1, w.d1, 1.f, nullptr, nullptr, nullptr, nullptr, nullptr, w.UTh, w.UTl, status, nullptr, w.UT3);
  launch_fold_split(st, V, w, w.Vh, w.Vl, w.V3, status);
  const uint16_t* a[3] = {w.UTh, w.UTl, w.UT3};
  const uint16_t* b[3] = {w.Vh, w.Vl, w.V3};
  DenseOut o;
  o.C = P; o.ldc = w.d3; o.Chi = w.Ph; o.Clo = w.Pl; o.Cthi = w.PTh; o.Ctlo = w.PTl;
  const int rc = launch_dense_tc(st, 3, a, 3, b, w.d1, w.d3, w.h, 1.f, 0.f, 0.f, o, P, status);
  if (rc) return rc;
  launch_split_rect(st, P, w.d1, w.d3, w.d3, 1.f, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, status, w.P3, w.PT3);
  return CAFEQ_OK;
}

// *sq += || Uhat_exp^T Vhat^T - P ||_F^2 ; optionally stores the residual R [d1, d3].  keep_splits: leaves the residual and its
// transpose in w.Ph / Pl / PTh / PTl and Uhat, as stored, in w.Awh / Awl (Vhat, replicas folded, is in w.Vh / Vl either way)
static int dense_pqe(cudaStream_t st, const float* Uhat, const float* Vhat, const float* P, DenseWS& w, double* sq, float* R,
                      int32_t* status, bool keep_splits = false) {
  launch_split_rect(st, Uhat, w.h, w.d1, w.d1, 1.f, nullptr, nullptr, nullptr, keep_splits ? w.Awh : nullptr,
                    keep_splits ? w.Awl : nullptr, w.UTh, w.UTl, status);
  launch_fold_split(st, Vhat, w, w.Vh, w.Vl, nullptr, status);
  const uint16_t* a[2] = {w.UTh, w.UTl};
  const uint16_t* b[2] = {w.Vh, w.Vl};
  DenseOut o;
  o.C0 = P; o.ldc0 = w.d3; o.C = R; o.ldc = w.d3; o.sq = sq;
  if (keep_splits) {  // the residual and its transpose as operands of the backward products
    o.Chi = w.Ph; o.Clo = w.Pl; o.Cthi = w.PTh; o.Ctlo = w.PTl;
  }
  return launch_dense_tc(st, 2, a, 2, b, w.d1, w.d3, w.h, 1.f, -1.f, 0.f, o, nullptr, status);
}

// Algorithm 1 on the transformed pair held in w.U [h, d1], w.V [d3, rh] (fp32, stored layout with r replicas of
// every inner block on the V side).  With E the replica expansion, the V update is Q((pinv((E Uhat)^T) P)^T) =
// Q(expand(pinv(Uhat^T) P) / r) (Uhat^T of full column rank) and the U update is Q((P pinv(fold(Vhat^T)))^T),
// which is the printed algorithm when r = 1.  pqe_hist: fp32 [2 iters + 1].
static int alg1_run(cudaStream_t st, int bits, int g1, int g2, int iters, int8_t* codes1, float* scales1, int8_t* codes2,
                     float* scales2, float* pqe_hist, DenseWS& w, int32_t* status) {
  int rc;
  CQ_LAUNCH(zero_f64_kernel, 1, 128, 0, st, w.sq, DENSE_SQ);
  if ((rc = dense_product(st, w.U, w.V, w, w.P, status))) return rc;
  quant_matrix(st, w.U, w.h, w.d1, g1, bits, codes1, scales1, w.Uhat, w, status);
  quant_matrix(st, w.V, w.d3, w.rh, g2, bits, codes2, scales2, w.Vhat, w, status);
  if ((rc = dense_pqe(st, w.Uhat, w.Vhat, w.P, w, w.sq + 0, nullptr, status))) return rc;
  for (int it = 0; it < iters; ++it) {
    // V side: X0^T [d3, h] = P^T pinv(Uhat^T)^T, then expand the replicas
    if ((rc = pinv_rows(st, w.Uhat, w.h, w.d1, w, status))) return rc;
    {
      const uint16_t* a[3] = {w.PTh, w.PTl, w.PT3};
      const uint16_t* b[3] = {w.Oh, w.Ol, w.O3};
      DenseOut o;
      o.C = w.X0T; o.ldc = w.h;
      if ((rc = launch_dense_tc(st, 3, a, 3, b, w.d3, w.h, w.d1, 1.f, 0.f, 0.f, o, w.X0T, status))) return rc;
    }
    CQ_LAUNCH(expand_cols_kernel, dim3(w.d3, (w.h + 1023) / 1024), 256, 0, st, w.X0T, w.h, w.k, w.r, 1.f / (float)w.r, w.V);
    quant_matrix(st, w.V, w.d3, w.rh, g2, bits, codes2, scales2, w.Vhat, w, status);
    if ((rc = dense_pqe(st, w.Uhat, w.Vhat, w.P, w, w.sq + 2 * it + 1, nullptr, status))) return rc;
    // U side: U' [h, d1] = pinv(Bf)^T P^T with Bf = fold(Vhat^T) [h, d3]
    {
      dim3 grid((w.d3 + 31) / 32, w.h / 32);
      CQ_LAUNCH(fold_transpose_kernel, grid, dim3(32, 8), 0, st, w.Vhat, w.d3, w.h, w.k, w.r, w.Bf);
    }
    if ((rc = pinv_rows(st, w.Bf, w.h, w.d3, w, status))) return rc;
    {
      const uint16_t* a[3] = {w.Oh, w.Ol, w.O3};
      const uint16_t* b[3] = {w.Ph, w.Pl, w.P3};
      DenseOut o;
      o.C = w.U; o.ldc = w.d1;
      if ((rc = launch_dense_tc(st, 3, a, 3, b, w.h, w.d1, w.d3, 1.f, 0.f, 0.f, o, w.U, status))) return rc;
    }
    quant_matrix(st, w.U, w.h, w.d1, g1, bits, codes1, scales1, w.Uhat, w, status);
    if ((rc = dense_pqe(st, w.Uhat, w.Vhat, w.P, w, w.sq + 2 * it + 2, nullptr, status))) return rc;
  }
  CQ_LAUNCH(sqrt_hist_kernel, 1, 128, 0, st, w.sq, pqe_hist, 2 * iters + 1);
  return CAFEQ_OK;
}

}  // namespace cafeq
