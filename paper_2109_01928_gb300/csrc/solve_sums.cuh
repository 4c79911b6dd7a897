// Mixed-precision weights, cost and gradient from the column sums, one thread per
// candidate: a kernel per pole count (pass_b*.cu), launched after its column-sum pass.
#pragma once
#include "common.cuh"

namespace debyefit {

// ------------------------------------------------------------------ cost from column sums (mixed)
// For the Debye columns c_i = 1/(1 + j w tau_i), partial fractions give
//   Re(c_i conj c_j) = (tau_i Re c_i + tau_j Re c_j) / (tau_i + tau_j),
// so the pole block of the Gram follows from the column sums S_i = sum_k re_i(k):
//   G_ij = (tau_i S_i + tau_j S_j) / (tau_i + tau_j),  G_ii = S_i  (re^2 + im^2 = re),
// and G_0i = S_i, G_00 = K for the eps_inf column. With h = A^T b and b^T b, the
// damped weights solve M x = h (M = G + lam diag G), and for the flipped x_hat
//   cost(x_hat) = b^T b - 2 x_hat^T h + x_hat^T M x_hat
// exactly. M, h, b^T b and the products with M are float-float (the subtraction
// loses the digits of b^T b / cost, about 4: float-float keeps ~9 of the ~13
// digits it carries); x comes from an FP32 Cholesky factor of the scaled M and
// refinement steps with the float-float residual h - M x.
constexpr int SUMS_REFINE = 2;       // refinement steps with the gradient (x and the adjoint w)
// Cost-only evaluations take one step: the scaled damped matrix C + lam I has unit
// diagonal, so kappa <= (n + lam) / lam (2e4 at n = 21, lam = 1e-3) and after one
// step the weights carry about (kappa 2^-24)^2 = 1.4e-6 relative error, which
// reaches a flipped candidate's cost at first order; two steps are ~2e-9.
constexpr int SUMS_REFINE_COST = 1;

__device__ __forceinline__ ff gram_ff(int i, int j, const ff* tau, const ff* S, ff kk) {
  if (i == 0 && j == 0) return kk;
  if (i == 0) return S[j - 1];
  if (j == 0 || i == j) return S[i - 1];
  const ff num = ff_sum(ff_prod(tau[i - 1], S[i - 1]), ff_prod(tau[j - 1], S[j - 1]));
  return ff_quot(num, ff_sum(tau[i - 1], tau[j - 1]));
}

// The float-float Gram entries (i >= j), formed where they are used (the compiler keeps
// what fits).
struct GramRecompute {
  const ff* tau;
  const ff* S;
  ff kk;
  __device__ __forceinline__ ff operator()(int i, int j) const { return gram_ff(i, j, tau, S, kk); }
};

// (M v)_i in float-float, M = G + lam diag G; each entry serves both of its rows.
template <class GA>
__device__ __forceinline__ void mvec_ff(int n, const GA& G, ff one_lam, const ff* v, ff* out) {
#pragma unroll
  for (int i = 0; i < n; ++i) out[i] = ff{0.f, 0.f};
#pragma unroll
  for (int i = 0; i < n; ++i) {
#pragma unroll
    for (int j = 0; j < i; ++j) {
      const ff g = G(i, j);
      out[i] = ff_sum(out[i], ff_prod(g, v[j]));
      out[j] = ff_sum(out[j], ff_prod(g, v[i]));
    }
    out[i] = ff_sum(out[i], ff_prod(ff_prod(G(i, i), one_lam), v[i]));
  }
}

// FP32 Cholesky L L^T of the scaled damped matrix, with 1 / L_jj stored on the
// diagonal so that the solves multiply instead of dividing.
template <class LA>
__device__ __forceinline__ bool cholesky_rdiag(LA L, int n) {
#pragma unroll
  for (int j = 0; j < n; ++j) {
    float s = L[pk(j, j)];
#pragma unroll
    for (int k = 0; k < j; ++k) s = __fmaf_rn(-L[pk(j, k)], L[pk(j, k)], s);
    if (!(s > 0.f) || !isfinite(s)) return false;
    const float inv = __frsqrt_rn(s);
    L[pk(j, j)] = inv;
#pragma unroll
    for (int i = j + 1; i < n; ++i) {
      float v = L[pk(i, j)];
#pragma unroll
      for (int k = 0; k < j; ++k) v = __fmaf_rn(-L[pk(i, k)], L[pk(j, k)], v);
      L[pk(i, j)] = __fmul_rn(v, inv);
    }
  }
  return true;
}

// v <- (L L^T)^-1 v for the factor of cholesky_rdiag
template <class LA>
__device__ __forceinline__ void llt_solve_rdiag(LA L, float* v, int n) {
#pragma unroll
  for (int i = 0; i < n; ++i) {
    float s = v[i];
#pragma unroll
    for (int k = 0; k < i; ++k) s = __fmaf_rn(-L[pk(i, k)], v[k], s);
    v[i] = __fmul_rn(s, L[pk(i, i)]);
  }
#pragma unroll
  for (int i = n - 1; i >= 0; --i) {
    float s = v[i];
#pragma unroll
    for (int k = i + 1; k < n; ++k) s = __fmaf_rn(-L[pk(k, i)], v[k], s);
    v[i] = __fmul_rn(s, L[pk(i, i)]);
  }
}

// M^-1 rhs through the FP32 factor L of the scaled M (scaling dinv = diag(G)^-1/2),
// refined `steps` times against the float-float M.
template <class LA, class GA>
__device__ __forceinline__ bool refined_solve(int n, LA L, const float* dinv, const GA& G, ff one_lam,
                                              const ff* rhs, ff* x, ff* r, float* v, int steps) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < n; ++i) x[i] = ff{0.f, 0.f};
#pragma unroll
  for (int it = 0; it <= steps && ok; ++it) {
    // r = rhs - M x (the first step has x = 0), dx = M^-1 r through the FP32 factor
    if (it == 0) {
#pragma unroll
      for (int i = 0; i < n; ++i) r[i] = rhs[i];
    } else {
      mvec_ff(n, G, one_lam, x, r);
#pragma unroll
      for (int i = 0; i < n; ++i) r[i] = ff_sum(rhs[i], ff_neg(r[i]));
    }
#pragma unroll
    for (int i = 0; i < n; ++i) v[i] = __fmul_rn(r[i].h, dinv[i]);
    llt_solve_rdiag(L, v, n);
#pragma unroll
    for (int i = 0; i < n; ++i) {
      x[i] = ff_sum(x[i], ff{__fmul_rn(v[i], dinv[i]), 0.f});
      ok = ok && isfinite(x[i].h);
    }
  }
  return ok;
}

// Cost (and, with grad, its derivative in theta) from the column sums. The
// gradient of cost(x_hat) = b^T b - 2 x_hat^T h + x_hat^T M x_hat, x_hat = s * x*
// (s the signs of the flip), x* = M^-1 h, is (variable projection with an
// adjoint for the flip)
//   d cost / d theta_i = -2 x_hat_i E_i + x_hat^T M_i x_hat + 2 (w_i E_i - w^T M_i x*),
//   w = M^-1 (s * (M x_hat - h)),
// with M_i = dM / d theta_i nonzero in row and column i only:
//   (M_i)_{i0} = D_i,  (M_i)_{ii} = (1 + lam) D_i,
//   (M_i)_{ij} = tau_i D_i / (tau_i + tau_j) + ln10 tau_i tau_j (S_i - S_j) / (tau_i + tau_j)^2
// (the derivative of G_ij = (tau_i S_i + tau_j S_j)/(tau_i + tau_j), d tau_i = ln10 tau_i).
//
// Every unit has NT poles (below SOLVE_ROLL_FROM; one launch per pole bucket): the loops
// unroll and the systems stay in registers. GRAD (0 or 1) fixes whether the gradient is
// computed.
template <int NT, int GRAD>
__global__ void __launch_bounds__(128) k_solve_sums_t(EvalArgs a, double* cost, double* weights, double* grad) {
  const int64_t Q = a.sc.Q;
  const int nmax = a.sc.nmax, nm1 = nmax + 1;
  constexpr bool with_grad = GRAD > 0;
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    const int q = u.q0 + (int)threadIdx.x;
    if (q >= u.q1 || (a.active && !a.active[q])) continue;
    if (u.N != NT) {
      set_status(a.status, DEBYE_EBOUNDS);
      continue;
    }
    constexpr int N = NT, n = N + 1;
    ff tau[N], S[N], hv[n], x[n], r[n];
    float L[n * (n + 1) / 2], dinv[n], v[n];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      tau[i] = load_ff(a.sc.x, (int64_t)i * Q + q);   // 10^theta_i from the column-sum pass
      S[i] = load_ff(a.sc.G, (int64_t)i * Q + q);
      hv[i + 1] = load_ff(a.sc.G, (int64_t)(N + i) * Q + q);
    }
    hv[0] = ff_of(a.h0[u.s]);
    const ff kk = ff_of_int((int)(u.k1 - u.k0));
    const ff one_lam = ff_of(1.0 + a.lam);
    const GramRecompute G{tau, S, kk};
    // FP32 Cholesky of the Marquardt-scaled damped matrix (unit diagonal + lam)
#pragma unroll
    for (int i = 0; i < n; ++i) dinv[i] = __frsqrt_rn(G(i, i).h);   // diag(G)^-1/2
#pragma unroll
    for (int i = 0; i < n; ++i) {
#pragma unroll
      for (int j = 0; j < i; ++j) L[pk(i, j)] = __fmul_rn(__fmul_rn(G(i, j).h, dinv[i]), dinv[j]);
      L[pk(i, i)] = (float)(1.0 + a.lam);
    }
    bool ok = cholesky_rdiag((float*)L, n);
    if (ok) ok = refined_solve(n, (float*)L, dinv, G, one_lam, hv, x, r, v, with_grad ? SUMS_REFINE : SUMS_REFINE_COST);
    record_fail(a, q, u.s, ok);
    if (!ok) {
      if (cost) cost[q] = INFINITY;
      if (weights)
        for (int j = 0; j < nm1; ++j) weights[(int64_t)q * nm1 + j] = 0.0;
      if (with_grad)
        for (int j = 0; j < nmax; ++j) grad[(int64_t)q * nmax + j] = 0.0;
      continue;
    }
    // sign flip of negative d_eps (Sec. III-B), then the exact quadratic cost
    float sgn[n];
#pragma unroll
    for (int i = 0; i < n; ++i) {
      sgn[i] = (i > 0 && x[i].h < 0.f) ? -1.f : 1.f;
      if (sgn[i] < 0.f) x[i] = ff_neg(x[i]);
    }
    mvec_ff(n, G, one_lam, x, r);   // r = M x_hat
    ff c = ff_of(a.bb[u.s]);
#pragma unroll
    for (int i = 0; i < n; ++i) {
      c = ff_sum(c, ff_neg(ff_prod(ff{__fmul_rn(2.f, x[i].h), __fmul_rn(2.f, x[i].l)}, hv[i])));
      c = ff_sum(c, ff_prod(x[i], r[i]));
    }
    double cv = ff_dbl(c);
    if (!isfinite(cv)) cv = INFINITY;
    if (cv < 0.0) cv = 0.0;
    if (cost) cost[q] = cv;
    if (weights) {
#pragma unroll
      for (int j = 0; j < n; ++j) weights[(int64_t)q * nm1 + j] = ff_dbl(x[j]);
      for (int j = n; j < nm1; ++j) weights[(int64_t)q * nm1 + j] = 0.0;
    }
    if (!with_grad) continue;
    // adjoint w = M^-1 (s * (M x_hat - h)); r becomes its right-hand side
    ff w[n], rw[n];
#pragma unroll
    for (int i = 0; i < n; ++i) {
      r[i] = ff_sum(r[i], ff_neg(hv[i]));
      if (sgn[i] < 0.f) r[i] = ff_neg(r[i]);
    }
    if (!refined_solve(n, (float*)L, dinv, G, one_lam, r, w, rw, v, SUMS_REFINE)) {
      for (int j = 0; j < nmax; ++j) grad[(int64_t)q * nmax + j] = 0.0;
      continue;
    }
    const ff ln10 = ff_of(2.302585092994046);
    for (int i = N; i < nmax; ++i) grad[(int64_t)q * nmax + i] = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int I = i + 1;
      const ff Di = load_ff(a.sc.G, (int64_t)(2 * N + i) * Q + q);
      const ff Ei = load_ff(a.sc.G, (int64_t)(3 * N + i) * Q + q);
      // row i of M_i against x_hat, w and x* (x*_j = s_j x_hat_j), off the diagonal
      ff ax = ff_prod(Di, x[0]), aw = ff_prod(Di, w[0]), as = ax;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        if (j == i) continue;
        const ff rr = ff_quot(ff{1.f, 0.f}, ff_sum(tau[i], tau[j]));
        const ff t1 = ff_prod(ff_prod(tau[i], Di), rr);
        const ff t2 = ff_prod(ff_prod(ff_prod(ln10, ff_prod(tau[i], tau[j])), ff_sum(S[i], ff_neg(S[j]))),
                              ff_prod(rr, rr));
        const ff row = ff_sum(t1, t2);
        const ff xs = sgn[j + 1] < 0.f ? ff_neg(x[j + 1]) : x[j + 1];
        ax = ff_sum(ax, ff_prod(row, x[j + 1]));
        aw = ff_sum(aw, ff_prod(row, w[j + 1]));
        as = ff_sum(as, ff_prod(row, xs));
      }
      const ff diag = ff_prod(Di, one_lam);
      const ff xhI = x[I], wI = w[I];
      const ff xsI = sgn[I] < 0.f ? ff_neg(xhI) : xhI;
      // x_hat^T M_i x_hat = 2 x_hat_i ax + diag x_hat_i^2;  w^T M_i x* = w_i as + x*_i aw + diag w_i x*_i
      ff gsum = ff_neg(ff_prod(ff{__fmul_rn(2.f, xhI.h), __fmul_rn(2.f, xhI.l)}, Ei));
      gsum = ff_sum(gsum, ff_prod(ff{__fmul_rn(2.f, xhI.h), __fmul_rn(2.f, xhI.l)}, ax));
      gsum = ff_sum(gsum, ff_prod(diag, ff_prod(xhI, xhI)));
      ff adj = ff_prod(wI, Ei);
      adj = ff_sum(adj, ff_neg(ff_prod(wI, as)));
      adj = ff_sum(adj, ff_neg(ff_prod(xsI, aw)));
      adj = ff_sum(adj, ff_neg(ff_prod(diag, ff_prod(wI, xsI))));
      gsum = ff_sum(gsum, ff{__fmul_rn(2.f, adj.h), __fmul_rn(2.f, adj.l)});
      grad[(int64_t)q * nmax + i] = ff_dbl(gsum);
    }
  }
}

// ------------------------------------------------------------------ rolled solve
// The same solve (operation for operation, so the same bits) for SOLVE_ROLL_FROM poles and
// more, with its code kept small: unrolled over all n^2 index pairs the float-float Gram
// entries and products take 13 000 instructions at N = 12, and with every warp of an SM
// streaming through that much code the instruction fetch bounds the kernel. Here the loops
// over rows stay loops; one row's columns are unrolled, so that the column operand (tau_j,
// p_j, x_j) sits in registers and the row's M entries come from shared memory, where they
// are formed once (packed lower triangle incl. row 0, diagonal already times 1 + lam). Only
// the FP32 factor, which is cheap per entry, is unrolled and held in registers. Two rows
// are in flight in the products with M: one float-float accumulation is a chain of 7
// dependent operations per term.
// One warp per block, one candidate per lane; element e of a lane's record at e * 32 + lane,
// so that a warp's 8-byte accesses are contiguous: 26.6 KB per block at N = 12 (8 blocks
// per SM), 64.5 KB at N = 20 (3; the factor then spills to L1). Measured on 65536 candidates, kernel timing, against the unrolled kernel: N = 12
// 229 -> 129 us, N = 8 75 -> 59 us, N = 4 31 -> 28 us (N = 3 equal, N = 2 slower, so the
// line lies at 4); with the gradient N = 12 1156 -> 368 us, N = 8 296 -> 167 us, N = 4
// 65 -> 56 us. With tau and the sums read in float-float instead of FP64: N = 12 86 us,
// N = 4 18 us, with the gradient 283 and 45 us. Against a general kernel with its arrays
// in local memory: N = 20 794 -> 522 us, N = 16 475 -> 221 us, with the gradient 1963 ->
// 1921 and 1283 -> 815 us.
constexpr int SOLVE_ROLL_FROM = 4;
constexpr int solve_roll_ff(int N) { return (N + 1) * (N + 2) / 2 + (N + 1); }   // M, then the product
constexpr size_t solve_roll_bytes(int N) { return sizeof(float2) * 32 * (size_t)solve_roll_ff(N); }

struct LaneFf {
  float2* p;
  __device__ __forceinline__ ff get(int e) const {
    const float2 v = p[e * 32];
    return ff{v.x, v.y};
  }
  __device__ __forceinline__ void put(int e, ff v) const { p[e * 32] = make_float2(v.h, v.l); }
};

// (M v)_i for all rows, into R: columns in ascending order, as mvec_ff accumulates them.
template <int n>
__device__ __forceinline__ void mvec_rows(const LaneFf& M, const LaneFf& R, const ff* v) {
#pragma unroll 1
  for (int i = 0; i < n; i += 2) {
    const int i1 = i + 1 < n ? i + 1 : i;   // the odd last row is formed twice
    const int b0 = pk(i, 0), b1 = pk(i1, 0);
    ff a0 = ff_prod(M.get(b0), v[0]), a1 = ff_prod(M.get(b1), v[0]);
#pragma unroll
    for (int j = 1; j < n; ++j) {
      const ff m0 = M.get(j <= i ? b0 + j : pk(j, 0) + i), m1 = M.get(j <= i1 ? b1 + j : pk(j, 0) + i1);
      a0 = ff_sum(a0, ff_prod(m0, v[j]));
      a1 = ff_sum(a1, ff_prod(m1, v[j]));
    }
    R.put(i, a0);
    R.put(i1, a1);
  }
}

// cholesky_rdiag and llt_solve_rdiag with every index known at compile time, so that the
// factor stays in registers.
template <int n>
__device__ __forceinline__ bool cholesky_regs(float (&L)[n * (n + 1) / 2]) {
  bool ok = true;
#pragma unroll
  for (int j = 0; j < n; ++j) {
    float s = L[pk(j, j)];
#pragma unroll
    for (int k = 0; k < n; ++k)
      if (k < j) s = __fmaf_rn(-L[pk(j, k)], L[pk(j, k)], s);
    ok = ok && s > 0.f && isfinite(s);
    const float inv = __frsqrt_rn(s);
    L[pk(j, j)] = inv;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      if (i <= j) continue;
      float v = L[pk(i, j)];
#pragma unroll
      for (int k = 0; k < n; ++k)
        if (k < j) v = __fmaf_rn(-L[pk(i, k)], L[pk(j, k)], v);
      L[pk(i, j)] = __fmul_rn(v, inv);
    }
  }
  return ok;
}

template <int n>
__device__ __forceinline__ void llt_solve_regs(const float (&L)[n * (n + 1) / 2], float (&v)[n]) {
#pragma unroll
  for (int i = 0; i < n; ++i) {
    float s = v[i];
#pragma unroll
    for (int k = 0; k < n; ++k)
      if (k < i) s = __fmaf_rn(-L[pk(i, k)], v[k], s);
    v[i] = __fmul_rn(s, L[pk(i, i)]);
  }
#pragma unroll
  for (int m = 0; m < n; ++m) {
    const int i = n - 1 - m;
    float s = v[i];
#pragma unroll
    for (int k = 0; k < n; ++k)
      if (k > i) s = __fmaf_rn(-L[pk(k, i)], v[k], s);
    v[i] = __fmul_rn(s, L[pk(i, i)]);
  }
}

// M^-1 rhs as refined_solve computes it.
template <int n>
__device__ __forceinline__ bool refined_solve_rows(const float (&L)[n * (n + 1) / 2], const float* dinv, const LaneFf& M,
                                                   const LaneFf& R, const ff* rhs, ff* x, int steps) {
  bool ok = true;
  float v[n];
#pragma unroll
  for (int i = 0; i < n; ++i) {
    x[i] = ff{0.f, 0.f};
    v[i] = __fmul_rn(rhs[i].h, dinv[i]);
  }
#pragma unroll 1
  for (int it = 0;; ++it) {
    llt_solve_regs<n>(L, v);
#pragma unroll
    for (int i = 0; i < n; ++i) {
      x[i] = ff_sum(x[i], ff{__fmul_rn(v[i], dinv[i]), 0.f});
      ok = ok && isfinite(x[i].h);
    }
    if (it == steps) break;
    mvec_rows<n>(M, R, x);
#pragma unroll
    for (int i = 0; i < n; ++i) v[i] = __fmul_rn(ff_sum(rhs[i], ff_neg(R.get(i))).h, dinv[i]);
  }
  return ok;
}

template <int N, int GRAD>
__global__ void __launch_bounds__(32) k_solve_rows(EvalArgs a, int slices, double* cost, double* weights,
                                                   double* grad) {
  constexpr int n = N + 1;
  extern __shared__ float2 solve_rows_smem[];
  const int64_t Q = a.sc.Q;
  const int nmax = a.sc.nmax, nm1 = nmax + 1;
  const LaneFf M{solve_rows_smem + threadIdx.x}, R{solve_rows_smem + threadIdx.x + 32 * pk(n, 0)};
  for (int ui = blockIdx.x; ui < a.n_units * slices; ui += gridDim.x) {
    const Unit u = a.units[ui / slices];
    const int q = u.q0 + ui % slices * 32 + (int)threadIdx.x;
    if (q >= u.q1 || (a.active && !a.active[q])) continue;
    if (u.N != N) {
      set_status(a.status, DEBYE_EBOUNDS);
      continue;
    }
    auto tau_of = [&](int i) { return load_ff(a.sc.x, (int64_t)i * Q + q); };
    auto S_of = [&](int i) { return load_ff(a.sc.G, (int64_t)i * Q + q); };
    const ff one_lam = ff_of(1.0 + a.lam);
    const ff kk = ff_of_int((int)(u.k1 - u.k0));
    float dinv[n];
    M.put(0, ff_prod(kk, one_lam));
    dinv[0] = __frsqrt_rn(kk.h);
    {
      // Gram entries, row by row: G_ij = (p_i + p_j) / (tau_i + tau_j), p = tau S
      ff tau[N], pr[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const ff S = S_of(i);
        tau[i] = tau_of(i);
        pr[i] = ff_prod(tau[i], S);
        dinv[i + 1] = __frsqrt_rn(S.h);
        M.put(pk(i + 1, 0), S);
        M.put(pk(i + 1, i + 1), ff_prod(S, one_lam));
      }
#pragma unroll 1
      for (int i = 1; i < N; ++i) {
        const ff ti = tau_of(i), pi = ff_prod(ti, M.get(pk(i + 1, 0)));
#pragma unroll
        for (int j0 = 0; j0 < N - 1; j0 += 4) {   // four independent quotients at a time
          if (j0 >= i) break;
          ff g[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int j = j0 + t;
            if (j < N - 1) g[t] = ff_quot(ff_sum(pi, pr[j]), ff_sum(ti, tau[j]));
          }
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int j = j0 + t;
            if (j < N - 1 && j < i) M.put(pk(i + 1, j + 1), g[t]);
          }
        }
      }
    }
    // FP32 Cholesky of the Marquardt-scaled damped matrix (unit diagonal + lam)
    float L[n * (n + 1) / 2];
#pragma unroll
    for (int i = 0; i < n; ++i) {
#pragma unroll
      for (int j = 0; j < i; ++j) L[pk(i, j)] = __fmul_rn(__fmul_rn(M.get(pk(i, j)).h, dinv[i]), dinv[j]);
      L[pk(i, i)] = (float)(1.0 + a.lam);
    }
    bool ok = cholesky_regs<n>(L);
    ff hv[n], x[n];
    hv[0] = ff_of(a.h0[u.s]);
#pragma unroll
    for (int i = 0; i < N; ++i) hv[i + 1] = load_ff(a.sc.G, (int64_t)(N + i) * Q + q);
    if (ok) ok = refined_solve_rows<n>(L, dinv, M, R, hv, x, GRAD ? SUMS_REFINE : SUMS_REFINE_COST);
    record_fail(a, q, u.s, ok);
    if (!ok) {
      if (cost) cost[q] = INFINITY;
      if (weights)
        for (int j = 0; j < nm1; ++j) weights[(int64_t)q * nm1 + j] = 0.0;
      if (GRAD)
        for (int j = 0; j < nmax; ++j) grad[(int64_t)q * nmax + j] = 0.0;
      continue;
    }
    // sign flip of negative d_eps (Sec. III-B), then the exact quadratic cost
    unsigned neg = 0;
#pragma unroll
    for (int i = 1; i < n; ++i)
      if (x[i].h < 0.f) {
        neg |= 1u << i;
        x[i] = ff_neg(x[i]);
      }
    mvec_rows<n>(M, R, x);   // R = M x_hat
    ff c = ff_of(a.bb[u.s]);
#pragma unroll
    for (int i = 0; i < n; ++i) {
      c = ff_sum(c, ff_neg(ff_prod(ff{__fmul_rn(2.f, x[i].h), __fmul_rn(2.f, x[i].l)}, hv[i])));
      c = ff_sum(c, ff_prod(x[i], R.get(i)));
    }
    double cv = ff_dbl(c);
    if (!isfinite(cv)) cv = INFINITY;
    if (cv < 0.0) cv = 0.0;
    if (cost) cost[q] = cv;
    if (weights) {
#pragma unroll
      for (int j = 0; j < n; ++j) weights[(int64_t)q * nm1 + j] = ff_dbl(x[j]);
      for (int j = n; j < nm1; ++j) weights[(int64_t)q * nm1 + j] = 0.0;
    }
    if constexpr (GRAD) {
      // adjoint w = M^-1 (s * (M x_hat - h)), its right-hand side in hv
      ff w[n];
#pragma unroll
      for (int i = 0; i < n; ++i) {
        hv[i] = ff_sum(R.get(i), ff_neg(hv[i]));
        if (neg >> i & 1u) hv[i] = ff_neg(hv[i]);
      }
      if (!refined_solve_rows<n>(L, dinv, M, R, hv, w, SUMS_REFINE)) {
        for (int j = 0; j < nmax; ++j) grad[(int64_t)q * nmax + j] = 0.0;
        continue;
      }
      const ff ln10 = ff_of(2.302585092994046);
      for (int i = N; i < nmax; ++i) grad[(int64_t)q * nmax + i] = 0.0;
      ff tau[N], S[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        tau[i] = tau_of(i);
        S[i] = M.get(pk(i + 1, 0));
        R.put(i + 1, w[i + 1]);
        M.put(i, x[i + 1]);   // rows 0 .. of M are free now: x_hat by index
      }
#pragma unroll 1
      for (int i = 0; i < N; ++i) {
        const int I = i + 1;
        const ff ti = tau_of(i), Si = S_of(i);
        const ff Di = load_ff(a.sc.G, (int64_t)(2 * N + i) * Q + q);
        const ff Ei = load_ff(a.sc.G, (int64_t)(3 * N + i) * Q + q);
        // row i of M_i against x_hat, w and x* (x*_j = s_j x_hat_j), off the diagonal
        ff ax = ff_prod(Di, x[0]), aw = ff_prod(Di, w[0]), as = ax;
#pragma unroll
        for (int j = 0; j < N; ++j) {
          if (j == i) continue;
          const ff rr = ff_quot(ff{1.f, 0.f}, ff_sum(ti, tau[j]));
          const ff t1 = ff_prod(ff_prod(ti, Di), rr);
          const ff t2 = ff_prod(ff_prod(ff_prod(ln10, ff_prod(ti, tau[j])), ff_sum(Si, ff_neg(S[j]))),
                                ff_prod(rr, rr));
          const ff row = ff_sum(t1, t2);
          const ff px = ff_prod(row, x[j + 1]);
          ax = ff_sum(ax, px);
          aw = ff_sum(aw, ff_prod(row, w[j + 1]));
          as = ff_sum(as, neg >> (j + 1) & 1u ? ff_neg(px) : px);
        }
        const ff diag = ff_prod(Di, one_lam);
        const ff xhI = M.get(i), wI = R.get(I);
        const ff xsI = neg >> I & 1u ? ff_neg(xhI) : xhI;
        // x_hat^T M_i x_hat = 2 x_hat_i ax + diag x_hat_i^2;  w^T M_i x* = w_i as + x*_i aw + diag w_i x*_i
        ff gsum = ff_neg(ff_prod(ff{__fmul_rn(2.f, xhI.h), __fmul_rn(2.f, xhI.l)}, Ei));
        gsum = ff_sum(gsum, ff_prod(ff{__fmul_rn(2.f, xhI.h), __fmul_rn(2.f, xhI.l)}, ax));
        gsum = ff_sum(gsum, ff_prod(diag, ff_prod(xhI, xhI)));
        ff adj = ff_prod(wI, Ei);
        adj = ff_sum(adj, ff_neg(ff_prod(wI, as)));
        adj = ff_sum(adj, ff_neg(ff_prod(xsI, aw)));
        adj = ff_sum(adj, ff_neg(ff_prod(diag, ff_prod(wI, xsI))));
        gsum = ff_sum(gsum, ff{__fmul_rn(2.f, adj.h), __fmul_rn(2.f, adj.l)});
        grad[(int64_t)q * nmax + i] = ff_dbl(gsum);
      }
    }
  }
}

}  // namespace debyefit
