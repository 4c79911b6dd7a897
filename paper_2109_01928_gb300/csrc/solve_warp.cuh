// Mixed-precision weights, cost and gradient from the column sums with one warp per
// candidate: at the end of the column-sum pass's units (eval.cuh) in small evaluations, or
// as a kernel of its own (kernels.cu).
#pragma once
#include "solve_sums.cuh"

namespace debyefit {

// ------------------------------------------------------------------ cost from column sums, a warp per candidate
// The algebra of solve_sums.cuh with lane r holding row r of the (N+1)-square
// systems, so that its O(N^2) loops run across the lanes: M one row per lane,
// the factorisation one column per step (rows in parallel), the triangular
// solves one unknown per step (broadcast by shuffle), the products with M one
// row per lane and the gradient one pole per lane. It serves evaluations too
// small to fill the GPU with one thread per candidate (the polish's line-search
// and accepted points), where a thread per candidate takes the latency of one candidate's
// serial solve: latency is all that bounds it. So each lane keeps its rows of M, L
// and L^T in registers (NP slots, the loops unrolled with a uniform exit at n) and
// every other lane's value comes by a shuffle that no earlier step delays: the
// factorisation updates all later columns at each step (its per-entry order, k
// ascending, is the one of the dot products), and the column an update broadcasts is
// the row of L^T its owner keeps. With M and L in shared memory, read entry by entry,
// the polish's 8192 points of 1024 spectra, N 2-12, with the gradient took 81 us (54
// now), one spectrum's 64 candidates of 3 poles 9 us (6).
constexpr unsigned FULL_MASK = 0xffffffffu;

__device__ __forceinline__ ff shfl_ff(ff v, int lane) {
  return ff{__shfl_sync(FULL_MASK, v.h, lane), __shfl_sync(FULL_MASK, v.l, lane)};
}

// Lane r's rows: M = G + lam diag G; the FP32 factor L of the scaled M, its columns
// (LT[j] = L_jr), and 1 / L_rr.
template <int NP>
struct WarpSystem {
  ff M[NP];
  float L[NP], LT[NP], dg;

  // L L^T = D^-1 M D^-1 in FP32 (the same operations as cholesky_rdiag)
  __device__ __forceinline__ bool factor(int n, int r) {
    dg = 0.f;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if (j >= n) break;
      const float s = __shfl_sync(FULL_MASK, L[j], j);
      if (!(s > 0.f) || !isfinite(s)) return false;
      const float inv = __frsqrt_rn(s);
      if (r == j) dg = inv;
      else L[j] = __fmul_rn(L[j], inv);
#pragma unroll
      for (int i = j + 1; i < NP; ++i) {
        if (i >= n) break;
        const float lij = __shfl_sync(FULL_MASK, L[j], i);
        if (r == j) LT[i] = lij;
        if (r >= i) L[i] = __fmaf_rn(-L[j], lij, L[i]);
      }
    }
    return true;
  }

  // (L L^T)^-1 b, lane r holding b_r and receiving the solution's entry r:
  // forward then backward substitution, one unknown per step.
  __device__ __forceinline__ float llt(int n, int r, float b) const {
    float acc = b, y = 0.f;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if (j >= n) break;
      const float yj = __shfl_sync(FULL_MASK, __fmul_rn(acc, dg), j);
      if (r == j) y = yj;
      if (r > j) acc = __fmaf_rn(-L[j], yj, acc);
    }
    acc = y;
    float x = 0.f;
#pragma unroll
    for (int jj = 0; jj < NP; ++jj) {
      const int j = NP - 1 - jj;
      if (j >= n) continue;
      const float xj = __shfl_sync(FULL_MASK, __fmul_rn(acc, dg), j);
      if (r == j) x = xj;
      if (r < j) acc = __fmaf_rn(-LT[j], xj, acc);
    }
    return x;
  }

  // (M v)_r, lane r holding v_r (zero for lanes r >= n)
  __device__ __forceinline__ ff mrow(int n, int r, ff v) const {
    ff acc{0.f, 0.f};
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if (j >= n) break;
      acc = ff_sum(acc, ff_prod(M[j], shfl_ff(v, j)));
    }
    return r < n ? acc : ff{0.f, 0.f};
  }

  // M^-1 rhs (lane r: rhs_r in, x_r out) through the FP32 factor (scaling di =
  // diag(G)^-1/2), refined `steps` times against the float-float M.
  __device__ __forceinline__ bool refined_solve(int n, int r, float di, ff rhs, ff& x, int steps) const {
    x = ff{0.f, 0.f};
    bool ok = true;
#pragma unroll 1
    for (int it = 0; it <= steps && ok; ++it) {
      ff res = rhs;
      if (it > 0) res = ff_sum(rhs, ff_neg(mrow(n, r, x)));
      const float dx = llt(n, r, __fmul_rn(res.h, di));
      x = ff_sum(x, ff{__fmul_rn(dx, di), 0.f});
      ok = __all_sync(FULL_MASK, r >= n || isfinite(x.h));
    }
    return ok;
  }
};

// Candidate q of unit u (q and the pole count the same in every lane; n = N + 1 <= NP).
template <int NP>
__device__ __forceinline__ void warp_solve(const EvalArgs& a, const Unit& u, int q, double* cost, double* weights,
                                           double* grad) {
  const int64_t Q = a.sc.Q;
  const int nmax = a.sc.nmax, nm1 = nmax + 1;
  const int r = (int)threadIdx.x & 31;
  const ff one_lam = ff_of(1.0 + a.lam);
  const int N = u.N, n = N + 1;
  // row r >= 1 is pole r - 1: tau (from the column-sum pass), S and h (and D, E)
  ff hv{0.f, 0.f}, S{0.f, 0.f}, tau{0.f, 0.f}, Di{0.f, 0.f}, Ei{0.f, 0.f};
  if (r == 0) {
    hv = ff_of(a.h0[u.s]);
    S = ff_of_int((int)(u.k1 - u.k0));   // G_00
  } else if (r < n) {
    tau = load_ff(a.sc.x, (int64_t)(r - 1) * Q + q);
    S = load_ff(a.sc.G, (int64_t)(r - 1) * Q + q);
    hv = load_ff(a.sc.G, (int64_t)(N + r - 1) * Q + q);
    if (grad) {
      Di = load_ff(a.sc.G, (int64_t)(2 * N + r - 1) * Q + q);
      Ei = load_ff(a.sc.G, (int64_t)(3 * N + r - 1) * Q + q);
    }
  }
  const float di = r < n ? __frsqrt_rn(S.h) : 0.f;
  const ff pr = ff_prod(tau, S);
  // row r of M and of the scaled FP32 matrix (unit diagonal + lam)
  WarpSystem<NP> m;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    m.M[j] = ff{0.f, 0.f};
    m.L[j] = m.LT[j] = 0.f;
    if (j >= n) continue;
    const ff Sj = shfl_ff(S, j), tj = shfl_ff(tau, j), pj = shfl_ff(pr, j);
    const float dj = __shfl_sync(FULL_MASK, di, j);
    ff g;
    if (j == 0 || j == r) g = S;
    else if (r == 0) g = Sj;
    else g = ff_quot(ff_sum(pr, pj), ff_sum(tau, tj));
    m.M[j] = j == r ? ff_prod(g, one_lam) : g;
    if (j < r) m.L[j] = __fmul_rn(__fmul_rn(g.h, di), dj);
    else if (j == r) m.L[j] = (float)(1.0 + a.lam);
  }
  bool ok = m.factor(n, r);
  ff x{0.f, 0.f};
  if (ok) ok = m.refined_solve(n, r, di, hv, x, grad ? SUMS_REFINE : SUMS_REFINE_COST);
  if (r == 0) record_fail(a, q, u.s, ok);
  if (!ok) {
    if (cost && r == 0) cost[q] = INFINITY;
    if (weights && r < nm1) weights[(int64_t)q * nm1 + r] = 0.0;
    if (grad && r < nmax) grad[(int64_t)q * nmax + r] = 0.0;
    return;
  }
  // sign flip of negative d_eps (Sec. III-B), then the exact quadratic cost
  const bool neg = r > 0 && r < n && x.h < 0.f;
  const unsigned flips = __ballot_sync(FULL_MASK, neg);
  if (neg) x = ff_neg(x);
  const ff mx = m.mrow(n, r, x);   // (M x_hat)_r
  const ff x2{__fmul_rn(2.f, x.h), __fmul_rn(2.f, x.l)};
  ff t{0.f, 0.f};
  if (r < n) t = ff_sum(ff_neg(ff_prod(x2, hv)), ff_prod(x, mx));
  for (int o = 16; o > 0; o >>= 1) t = ff_sum(t, ff{__shfl_xor_sync(FULL_MASK, t.h, o),
                                                    __shfl_xor_sync(FULL_MASK, t.l, o)});
  if (r == 0 && cost) {
    double cv = ff_dbl(ff_sum(ff_of(a.bb[u.s]), t));
    if (!isfinite(cv)) cv = INFINITY;
    if (cv < 0.0) cv = 0.0;
    cost[q] = cv;
  }
  if (weights && r < nm1) weights[(int64_t)q * nm1 + r] = r < n ? ff_dbl(x) : 0.0;
  if (!grad) return;
  // adjoint w = M^-1 (s * (M x_hat - h))
  ff rw{0.f, 0.f};
  if (r < n) {
    rw = ff_sum(mx, ff_neg(hv));
    if (neg) rw = ff_neg(rw);
  }
  ff w;
  if (!m.refined_solve(n, r, di, rw, w, SUMS_REFINE)) {
    if (r < nmax) grad[(int64_t)q * nmax + r] = 0.0;
    return;
  }
  // d cost / d theta_i in lane r = i + 1 (the formula in solve_sums.cuh)
  const ff ln10 = ff_of(2.302585092994046);
  ff ax = ff_prod(Di, shfl_ff(x, 0)), aw = ff_prod(Di, shfl_ff(w, 0)), as = ax;
#pragma unroll
  for (int j = 1; j < NP; ++j) {
    if (j >= n) break;
    const ff tj = shfl_ff(tau, j), Sj = shfl_ff(S, j), xj = shfl_ff(x, j), wj = shfl_ff(w, j);
    if (j == r) continue;
    const ff rr = ff_quot(ff{1.f, 0.f}, ff_sum(tau, tj));
    const ff t1 = ff_prod(ff_prod(tau, Di), rr);
    const ff t2 = ff_prod(ff_prod(ff_prod(ln10, ff_prod(tau, tj)), ff_sum(S, ff_neg(Sj))), ff_prod(rr, rr));
    const ff row = ff_sum(t1, t2);
    const ff px = ff_prod(row, xj);
    ax = ff_sum(ax, px);
    aw = ff_sum(aw, ff_prod(row, wj));
    as = ff_sum(as, flips >> j & 1u ? ff_neg(px) : px);
  }
  if (r >= 1 && r <= nmax) {
    double gi = 0.0;
    if (r < n) {
      const ff diag = ff_prod(Di, one_lam);
      const ff xsI = neg ? ff_neg(x) : x;
      ff gsum = ff_neg(ff_prod(x2, Ei));
      gsum = ff_sum(gsum, ff_prod(x2, ax));
      gsum = ff_sum(gsum, ff_prod(diag, ff_prod(x, x)));
      ff adj = ff_prod(w, Ei);
      adj = ff_sum(adj, ff_neg(ff_prod(w, as)));
      adj = ff_sum(adj, ff_neg(ff_prod(xsI, aw)));
      adj = ff_sum(adj, ff_neg(ff_prod(diag, ff_prod(w, xsI))));
      gsum = ff_sum(gsum, ff{__fmul_rn(2.f, adj.h), __fmul_rn(2.f, adj.l)});
      gi = ff_dbl(gsum);
    }
    grad[(int64_t)q * nmax + r - 1] = gi;
  }
}

}  // namespace debyefit
