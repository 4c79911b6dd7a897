// N-generic kernels of libdebyefit: input preparation, the FP64 damped solve,
// refinement/finish with the sign flip, gradient assembly, the particle swarm
// and target synthesis.
#include <cmath>

#include "launch.h"
#include "solve.cuh"
#include "solve_warp.cuh"

namespace debyefit {

// ------------------------------------------------------------------ input preparation
// Per sample: float-float splits of (omega 2^-30)^2, eps' and omega eps'' for the column
// sums (the planes of EvalArgs), and finiteness checks; per spectrum: the granules, h0 =
// sum_k eps'_k and b^T b (FP64).
struct PrepPlanes {
  float4 *kq0, *kq1, *kq2;
};
struct PrepSample {
  ff w2, e, c;
  __device__ __forceinline__ PrepSample(double w, double a, double b, int* status) {
    if (!(w > 0.0) || !isfinite(w) || !isfinite(a) || !isfinite(b)) set_status(status, DEBYE_ENOTFINITE);
    const double ws = w * 0x1p-30;
    w2 = ff_of(ws * ws);
    e = ff_of(a);
    c = ff_of(w * b);
  }
  __device__ __forceinline__ void write(const PrepPlanes& p, int64_t k) const {
    p.kq0[k] = make_float4(w2.h, w2.h, w2.l, w2.l);
    p.kq1[k] = make_float4(e.h, e.h, e.l, e.l);
    p.kq2[k] = make_float4(c.h, c.h, c.l, c.l);
  }
};

// The bounds of a granule, a sample per lane: {smallest (omega 2^-30)^2, largest eps', largest
// omega eps'', largest (omega 2^-30)^2}.
struct PrepGranule {
  float w2lo = INFINITY, w2hi = 0.f, e = 0.f, c = 0.f;   // neutral for the lanes past the spectrum's end
  __device__ __forceinline__ void take(const PrepSample& smp) {
    w2lo = w2hi = smp.w2.h;   // the factor of the bounds' test covers its rounding
    e = smp.e.h;
    c = smp.c.h;
    if (!(e >= 0.f && e < INFINITY && c >= 0.f && c < INFINITY && w2lo >= 0.f)) e = c = INFINITY;
  }
  __device__ __forceinline__ void write(float4* at) {
    for (int o = 16; o > 0; o >>= 1) {
      w2lo = fminf(w2lo, __shfl_xor_sync(0xffffffffu, w2lo, o));
      w2hi = fmaxf(w2hi, __shfl_xor_sync(0xffffffffu, w2hi, o));
      e = fmaxf(e, __shfl_xor_sync(0xffffffffu, e, o));
      c = fmaxf(c, __shfl_xor_sync(0xffffffffu, c, o));
    }
    if ((threadIdx.x & 31) == 0) *at = make_float4(w2lo, e, c, w2hi);
  }
};
static_assert(GRANULE == 32, "a granule is a warp's samples");

// Planes and granules, PREP_RUN places of kg a warp's turn: the spectrum of the first is found
// by bisection of the spectra's first places (they ascend), the others follow. Spread over
// the whole grid whatever the spectra's lengths.
constexpr int PREP_RUN = 4;
__global__ void k_prep_samples(int64_t places, int64_t S, const int64_t* __restrict__ offsets,
                               const double* __restrict__ omega, const double* __restrict__ er,
                               const double* __restrict__ ei, float4* __restrict__ kg, PrepPlanes planes, int* status) {
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = (int64_t)gridDim.x * blockDim.x >> 5;
  for (int64_t g0 = warp * PREP_RUN; g0 < places; g0 += warps * PREP_RUN) {
    int64_t s = 0, last = S - 1;
    while (s < last) {
      const int64_t m = (s + last + 1) >> 1;
      if (granule_base(offsets[m], m) <= g0) s = m;
      else last = m - 1;
    }
    for (int64_t g = g0; g < g0 + PREP_RUN && g < places; ++g) {
      while (s + 1 < S && granule_base(offsets[s + 1], s + 1) <= g) ++s;
      const int64_t a = offsets[s], b = offsets[s + 1], k0 = a + (g - granule_base(a, s)) * GRANULE;
      if (k0 >= b) continue;   // a place that the spectrum does not fill
      const int64_t k = k0 + (threadIdx.x & 31);
      PrepGranule gr;
      if (k < b) {
        const PrepSample smp(omega[k], er[k], ei[k], status);
        smp.write(planes, k);
        gr.take(smp);
      }
      gr.write(kg + g);
    }
  }
}

// h0 and b^T b, one block per spectrum. MERGED: the planes and granules too (each warp's 32
// samples of an iteration are one granule), one launch and one read of the samples for both.
// A long spectrum's would be one block's work: there k_prep_samples makes them.
template <bool MERGED>
__global__ void k_prep_spectra(int64_t S, const int64_t* __restrict__ offsets, const double* __restrict__ omega,
                               const double* __restrict__ er, const double* __restrict__ ei,
                               const double* __restrict__ lo, const double* __restrict__ hi,
                               double* __restrict__ h0, double* __restrict__ bb, float4* __restrict__ kg,
                               PrepPlanes planes, int* status) {
  __shared__ double red[32], red2[32];
  for (int64_t s = blockIdx.x; s < S; s += gridDim.x) {
    const int64_t a = offsets[s], b = offsets[s + 1];
    double acc = 0.0, acc2 = 0.0;
    if constexpr (!MERGED) {
      for (int64_t k = a + threadIdx.x; k < b; k += blockDim.x) {
        acc += er[k];
        acc2 = fma(er[k], er[k], fma(ei[k], ei[k], acc2));
      }
    } else {
      for (int64_t k0 = a + (threadIdx.x & ~31u); k0 < b; k0 += blockDim.x) {
        const int64_t k = k0 + (threadIdx.x & 31);
        PrepGranule gr;
        if (k < b) {
          const double r = er[k], i = ei[k];
          acc += r;
          acc2 = fma(r, r, fma(i, i, acc2));
          const PrepSample smp(omega[k], r, i, status);
          smp.write(planes, k);
          gr.take(smp);
        }
        gr.write(kg + granule_base(a, s) + (k0 - a) / GRANULE);
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      acc += __shfl_down_sync(0xffffffffu, acc, o);
      acc2 += __shfl_down_sync(0xffffffffu, acc2, o);
    }
    if ((threadIdx.x & 31) == 0) {
      red[threadIdx.x >> 5] = acc;
      red2[threadIdx.x >> 5] = acc2;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      acc = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
      acc2 = (threadIdx.x < (blockDim.x >> 5)) ? red2[threadIdx.x] : 0.0;
      for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_down_sync(0xffffffffu, acc, o);
        acc2 += __shfl_down_sync(0xffffffffu, acc2, o);
      }
      if (threadIdx.x == 0) {
        h0[s] = acc;
        bb[s] = acc2;
        if (!(lo[s] < hi[s]) || !isfinite(lo[s]) || !isfinite(hi[s])) set_status(status, DEBYE_EBOUNDS);
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ damped solve
// Scaling helpers of the factor type T: in FP64 a division by d = 1/dinv (as the
// plain method reads); in FP32 a multiplication by dinv.
template <typename T>
struct Scale {
  T dinv[NMAX1];   // 1 / sqrt(G_ii)
  double d[NMAX1]; // sqrt(G_ii)
  __device__ __forceinline__ void load(const Scratch& sc, int64_t q, int n) {
    for (int i = 0; i < n; ++i) {
      dinv[i] = (T)sc.dinv[(int64_t)i * sc.Q + q];
      if constexpr (sizeof(T) == 8) d[i] = 1.0 / sc.dinv[(int64_t)i * sc.Q + q];
      else d[i] = (double)(1.0f / dinv[i]);
    }
  }
  // D^-1 v for an FP64 vector entry, as T
  __device__ __forceinline__ T down(double v, int i) const {
    if constexpr (sizeof(T) == 8) return v / d[i];
    else return (float)v * dinv[i];
  }
  // D^-1 v for a T entry, as FP64
  __device__ __forceinline__ double up(T v, int i) const {
    if constexpr (sizeof(T) == 8) return v / d[i];
    else return (double)(v * dinv[i]);
  }
};

// x0 = M^-1 h per candidate; stores L (type T), D^-1, x0 and the failure flag.
template <typename T>
__global__ void __launch_bounds__(256) k_solve(EvalArgs a) {
  const int64_t Q = a.sc.Q;
  const int hb = (a.sc.nmax + 1) * (a.sc.nmax + 2) / 2;
  T* Lg = factor_base_w<T>(a.sc);
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    const int q = u.q0 + (int)threadIdx.x;
    if (q >= u.q1 || (a.active && !a.active[q])) continue;
    const int n = u.N + 1;
    T L[NPACK_MAX], dinv[NMAX1], z[NMAX1];
    for (int i = 0; i < n; ++i) dinv[i] = T(1) / sqrt_t((T)a.sc.G[(int64_t)pk(i, i) * Q + q]);
    for (int i = 0; i < n; ++i) {
      for (int j = 0; j < i; ++j) L[pk(i, j)] = (T)a.sc.G[(int64_t)pk(i, j) * Q + q] * dinv[i] * dinv[j];
      L[pk(i, i)] = (T)(1.0 + a.lam);
    }
    bool ok = cholesky_packed(L, n);
    double x0[NMAX1];
    if (ok) {
      for (int i = 0; i < n; ++i) z[i] = (T)a.sc.G[(int64_t)(hb + i) * Q + q] * dinv[i];
      llt_solve(L, z, n);
      for (int i = 0; i < n; ++i) {
        x0[i] = (double)(z[i] * dinv[i]);
        ok = ok && isfinite(x0[i]);
      }
    }
    record_fail(a, q, u.s, ok);
    if (!ok) continue;
    const int npk = n * (n + 1) / 2;
    for (int e = 0; e < npk; ++e) Lg[(int64_t)e * Q + q] = L[e];
    for (int i = 0; i < n; ++i) {
      a.sc.dinv[(int64_t)i * Q + q] = (double)dinv[i];
      a.sc.x[(int64_t)i * Q + q] = x0[i];
    }
  }
}

// ------------------------------------------------------------------ refinement / finish
// From the residual pass at x (rt: rr = ||b - A x||^2, t = A^T (b - A x)):
//   g  = t - lam diag(G) x          (minus half the cost gradient in x)
//   dx = M^-1 g,  x1 = x + dx       (one step of iterative refinement)
// final == 0: store x1 and return.
// final == 1: cost(x1) by the exact quadratic identity
//   cost(y) = cost(x) - 2 (y - x)^T g + (y - x)^T M (y - x),  cost(x) = rr + lam sum G_ii x_i^2,
// then the sign flip x_hat = x1 + e (e_i = -2 x1_i where d_eps_i < 0, Sec. III-B) and
//   cost(x_hat) = cost(x1) - 2 e^T g1 + e^T M e,  g1 = g - M dx.
// Outputs cost[q], weights[q][nmax+1] (optional); keeps x1, x_hat and g1 for the gradient.
// Sums of the cost identity are FP64; products with the factor are in its type T.
template <typename T>
__global__ void __launch_bounds__(256) k_finish(EvalArgs a, int final_step, double* cost,
                                                double* weights, double* g1_out) {
  const int64_t Q = a.sc.Q;
  const int nm1 = a.sc.nmax + 1;
  const T* Lg = factor_base<T>(a.sc);
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    const int q = u.q0 + (int)threadIdx.x;
    if (q >= u.q1 || (a.active && !a.active[q])) continue;
    const int n = u.N + 1;
    if (a.sc.fail[q]) {
      if (final_step) {
        if (cost) cost[q] = INFINITY;
        if (weights)
          for (int j = 0; j < nm1; ++j) weights[(int64_t)q * nm1 + j] = 0.0;
      }
      continue;
    }
    T L[NPACK_MAX], v[NMAX1], w1[NMAX1], tmp[NMAX1];
    double x[NMAX1], g[NMAX1], dx[NMAX1];
    Scale<T> sc;
    sc.load(a.sc, q, n);
    const int npk = n * (n + 1) / 2;
    for (int e = 0; e < npk; ++e) L[e] = Lg[(int64_t)e * Q + q];
    double cost0 = a.sc.rt[q];
    for (int i = 0; i < n; ++i) {
      const double gii = a.sc.G[(int64_t)pk(i, i) * Q + q];
      x[i] = a.sc.x[(int64_t)i * Q + q];
      g[i] = a.sc.rt[(int64_t)(i + 1) * Q + q] - a.lam * gii * x[i];
      cost0 += a.lam * gii * x[i] * x[i];
      v[i] = sc.down(g[i], i);
    }
    llt_solve(L, v, n);            // v = D dx
    for (int i = 0; i < n; ++i) dx[i] = sc.up(v[i], i);
    if (!final_step) {
      for (int i = 0; i < n; ++i) a.sc.x[(int64_t)i * Q + q] = x[i] + dx[i];
      continue;
    }
    lt_mul(L, v, w1, n);           // w1 = L^T D dx
    double dg = 0.0, dmd = 0.0;
    for (int i = 0; i < n; ++i) {
      dg += dx[i] * g[i];
      dmd += (double)w1[i] * (double)w1[i];
    }
    double c = cost0 - 2.0 * dg + dmd;
    // The step must not raise the damped cost, whose value at x is exact: if the
    // identity leaves [0, cost(x)] the refinement is discarded (dx = 0).
    if (!(c >= 0.0 && c <= cost0)) {
      c = cost0;
      for (int i = 0; i < n; ++i) {
        dx[i] = 0.0;
        w1[i] = T(0);
      }
    }
    l_mul(L, w1, tmp, n);          // tmp = L L^T D dx; M dx = D tmp
    bool flipped = false;
    double e[NMAX1];
    for (int i = 0; i < n; ++i) {
      const double x1 = x[i] + dx[i];
      x[i] = x1;
      g[i] -= sc.d[i] * (double)tmp[i];   // g1
      e[i] = (i > 0 && x1 < 0.0) ? -2.0 * x1 : 0.0;
      flipped |= (e[i] != 0.0);
    }
    if (flipped) {
      for (int i = 0; i < n; ++i) tmp[i] = (T)(sc.d[i] * e[i]);
      lt_mul(L, tmp, w1, n);
      double eg = 0.0, eme = 0.0;
      for (int i = 0; i < n; ++i) {
        eg += e[i] * g[i];
        eme += (double)w1[i] * (double)w1[i];
      }
      c = c - 2.0 * eg + eme;
    }
    if (!isfinite(c)) c = INFINITY;
    if (cost) cost[q] = c;
    for (int i = 0; i < n; ++i) {
      a.sc.x[(int64_t)i * Q + q] = x[i];
      a.sc.xh[(int64_t)i * Q + q] = x[i] + e[i];
      if (g1_out) g1_out[(int64_t)i * Q + q] = g[i];
    }
    if (weights) {
      for (int j = 0; j < nm1; ++j) weights[(int64_t)q * nm1 + j] = (j < n) ? x[j] + e[j] : 0.0;
    }
  }
}

constexpr int WARP_SOLVE_WARPS = 4;         // candidates per block
constexpr int WARP_SOLVE_MAX_Q_PER_SM = 256; // auto choice: at most this many candidates per SM

// (4 resident blocks only where they cost no spills: at 21 slots 25 us against 33 for 61 x 37
// candidates; at 13 slots any such bound gave 75 us against 66 for 1024 x 8 points.)
template <int NP>
__global__ void __launch_bounds__(WARP_SOLVE_WARPS * 32, (NP > 13 ? 4 : 0)) k_solve_sums_warp(EvalArgs a, int slices, double* cost,
                                                                           double* weights, double* grad) {
  const int wid = (int)threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  for (int ui = blockIdx.x; ui < a.n_units * slices; ui += gridDim.x) {
    const Unit u = a.units[ui / slices];
    const int q = u.q0 + ui % slices * nw + wid;   // warp-uniform
    if (q >= u.q1 || (a.active && !a.active[q])) continue;
    if (u.N >= NP) {
      set_status(a.status, DEBYE_EBOUNDS);
      continue;
    }
    warp_solve<NP>(a, u, q, cost, weights, grad);
  }
}

// ------------------------------------------------------------------ gradient
// w = M^-1 S g_hat with g_hat = g1 - M (x_hat - x1) = h - M x_hat,
// S = diag(1, sign x1_1, ..., sign x1_N).
template <typename T>
__global__ void __launch_bounds__(256) k_grad_prep(EvalArgs a, const double* g1, double* sg_out) {
  const int64_t Q = a.sc.Q;
  const T* Lg = factor_base<T>(a.sc);
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    const int q = u.q0 + (int)threadIdx.x;
    if (q >= u.q1 || (a.active && !a.active[q])) continue;
    if (a.sc.fail[q]) continue;
    const int n = u.N + 1;
    T L[NPACK_MAX], t1[NMAX1], t2[NMAX1];
    double e[NMAX1];
    Scale<T> sc;
    sc.load(a.sc, q, n);
    const int npk = n * (n + 1) / 2;
    for (int k = 0; k < npk; ++k) L[k] = Lg[(int64_t)k * Q + q];
    for (int i = 0; i < n; ++i) {
      const double x1 = a.sc.x[(int64_t)i * Q + q];
      e[i] = a.sc.xh[(int64_t)i * Q + q] - x1;
      t1[i] = (T)(sc.d[i] * e[i]);
    }
    lt_mul(L, t1, t2, n);
    l_mul(L, t2, t1, n);           // M e = D t1
    for (int i = 0; i < n; ++i) {
      const double x1 = a.sc.x[(int64_t)i * Q + q];
      double gh = g1[(int64_t)i * Q + q] - sc.d[i] * (double)t1[i];
      if (i > 0 && x1 < 0.0) gh = -gh;
      if (sg_out) sg_out[(int64_t)i * Q + q] = gh;   // S g_hat, kept for the refinement of w
      t2[i] = sc.down(gh, i);
    }
    llt_solve(L, t2, n);
    for (int i = 0; i < n; ++i) a.sc.w[(int64_t)i * Q + q] = sc.up(t2[i], i);
  }
}

__global__ void __launch_bounds__(256) k_grad_finish(EvalArgs a, double* grad) {
  const int64_t Q = a.sc.Q;
  const int nmax = a.sc.nmax;
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    const int q = u.q0 + (int)threadIdx.x;
    if (q >= u.q1 || (a.active && !a.active[q])) continue;
    const int N = u.N;
    if (a.sc.fail[q]) {
      for (int i = 0; i < nmax; ++i) grad[(int64_t)q * nmax + i] = 0.0;
      continue;
    }
    for (int i = 0; i < nmax; ++i) {
      double gi = 0.0;
      if (i < N) {
        const double xh = a.sc.xh[(int64_t)(i + 1) * Q + q];
        const double x1 = a.sc.x[(int64_t)(i + 1) * Q + q];
        const double w = a.sc.w[(int64_t)(i + 1) * Q + q];
        const double t_rh = a.sc.gt[(int64_t)i * Q + q];
        const double t_aa = a.sc.gt[(int64_t)(N + i) * Q + q];
        const double t_r = a.sc.gt[(int64_t)(2 * N + i) * Q + q];
        const double t_aw = a.sc.gt[(int64_t)(3 * N + i) * Q + q];
        gi = -2.0 * xh * t_rh + 2.0 * a.lam * xh * xh * t_aa - 2.0 * w * t_r +
             4.0 * a.lam * w * x1 * t_aa + 2.0 * x1 * t_aw;
      }
      grad[(int64_t)q * nmax + i] = gi;
    }
  }
}

// ------------------------------------------------------------------ host launchers
void launch_prep(int64_t n_samples, int64_t S, int64_t longest, const int64_t* offsets, const double* omega,
                 const double* er, const double* ei, const double* lo, const double* hi,
                 float4* kq0, float4* kq1, float4* kq2, float4* kg, double* h0, int* status, int sms,
                 cudaStream_t st) {
  const PrepPlanes planes{kq0, kq1, kq2};
  if (S <= 0) return;
  const int grid = (int)std::min<int64_t>(S, (int64_t)sms * 8);
  if (prep_merged(longest)) {
    k_prep_spectra<true><<<grid, 256, 0, st>>>(S, offsets, omega, er, ei, lo, hi, h0, h0 + S, kg, planes, status);
    return;
  }
  const int64_t places = granule_count(n_samples, S), per_block = 8 * PREP_RUN;
  const int sgrid = (int)std::min<int64_t>((places + per_block - 1) / per_block, (int64_t)sms * 16);
  k_prep_samples<<<sgrid, 256, 0, st>>>(places, S, offsets, omega, er, ei, kg, planes, status);
  k_prep_spectra<false><<<grid, 256, 0, st>>>(S, offsets, omega, er, ei, lo, hi, h0, h0 + S, kg, planes, status);
}

static int grid_for(int n_units, int sms, int per_sm) {
  return std::max(1, std::min(n_units, sms * per_sm));
}

bool solve_sums_by_warp(int64_t Q, int lanes, int sms) {
  if (lanes == 1 || lanes == 32) return lanes == 32;
  return Q <= (int64_t)sms * WARP_SOLVE_MAX_Q_PER_SM;
}

// Blocks of up to 4 warps, one candidate each. The batch's pole capacity picks the number
// of slots, so that one launch after the join serves every pole count of it (a launch per
// pole count behind its pass measured slower: 1024 spectra x 8 points with the gradient, 299
// us against 286).
void launch_solve_sums_warp(const EvalArgs& a, double* cost, double* weights, double* grad, int cands_per_unit,
                            int sms, cudaStream_t st) {
  if (!a.n_units) return;
  const int warps = std::max(1, std::min(WARP_SOLVE_WARPS, cands_per_unit));
  const int slices = (cands_per_unit + warps - 1) / warps;
  const int grid = (int)std::min<int64_t>((int64_t)a.n_units * slices, (int64_t)sms * 64);
  const int n1 = a.sc.nmax + 1;
  if (n1 <= 5) k_solve_sums_warp<5><<<grid, warps * 32, 0, st>>>(a, slices, cost, weights, grad);
  else if (n1 <= 9) k_solve_sums_warp<9><<<grid, warps * 32, 0, st>>>(a, slices, cost, weights, grad);
  else if (n1 <= 13) k_solve_sums_warp<13><<<grid, warps * 32, 0, st>>>(a, slices, cost, weights, grad);
  else k_solve_sums_warp<NMAX1><<<grid, warps * 32, 0, st>>>(a, slices, cost, weights, grad);
}

void launch_solve(const EvalArgs& a, int block, int sms, cudaStream_t st) {
  if (a.n_units) k_solve<double><<<grid_for(a.n_units, sms, 8), block, 0, st>>>(a);
}
void launch_finish(const EvalArgs& a, int final_step, double* cost, double* weights, double* g1,
                   int block, int sms, cudaStream_t st) {
  if (a.n_units) k_finish<double><<<grid_for(a.n_units, sms, 8), block, 0, st>>>(a, final_step, cost, weights, g1);
}
void launch_grad_prep(const EvalArgs& a, const double* g1, double* sg_out, int block, int sms, cudaStream_t st) {
  if (a.n_units) k_grad_prep<double><<<grid_for(a.n_units, sms, 8), block, 0, st>>>(a, g1, sg_out);
}
void launch_grad_finish(const EvalArgs& a, double* grad, int block, int sms, cudaStream_t st) {
  if (a.n_units) k_grad_finish<<<grid_for(a.n_units, sms, 8), block, 0, st>>>(a, grad);
}

}  // namespace debyefit

// ------------------------------------------------------------------ target synthesis (Eqs. 3-7)
namespace debyefit {

struct cplx {
  double re, im;
};
__device__ __forceinline__ cplx c_add(cplx a, cplx b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cplx c_scale(cplx a, double s) { return {a.re * s, a.im * s}; }
// Principal power z^p = |z|^p exp(j p arg z).
__device__ __forceinline__ cplx c_pow(cplx z, double p) {
  const double m = pow(hypot(z.re, z.im), p), t = p * atan2(z.im, z.re);
  double sn, cs;
  sincos(t, &sn, &cs);
  return {m * cs, m * sn};
}
// Debye pole eps_inf + d_eps / (1 + j x), x = omega tau (Eq. 3), as a complex number.
__device__ __forceinline__ cplx c_debye(double ei, double de, double x) {
  const double r = 1.0 / (1.0 + x * x);
  return {ei + de * r, -de * x * r};
}

__global__ void k_synth(int64_t S, const int64_t* __restrict__ offsets, const double* __restrict__ omega,
                        const int32_t* __restrict__ model, const double* __restrict__ params,
                        const int64_t* __restrict__ pole_off, const double* __restrict__ ptau,
                        const double* __restrict__ pdeps, const double* __restrict__ nre,
                        const double* __restrict__ nim, double* __restrict__ er,
                        double* __restrict__ ei, int* status) {
  constexpr double PI = 3.141592653589793;
  for (int64_t s = blockIdx.x; s < S; s += gridDim.x) {
    const double* p = params + s * DEBYE_N_PARAMS;
    const int m = model[s];
    for (int64_t k = offsets[s] + threadIdx.x; k < offsets[s + 1]; k += blockDim.x) {
      const double w = omega[k];
      cplx e = {0.0, 0.0};
      double sigma = 0.0;
      switch (m) {
        case DEBYE_MODEL_DEBYE:
          e = c_debye(p[0], p[1], w * p[2]);
          break;
        case DEBYE_MODEL_HN:
        case DEBYE_MODEL_CC:
        case DEBYE_MODEL_CD: {
          // (j w tau0)^alpha on the principal branch, then (1 + .)^beta
          const double al = p[3], be = p[4];
          const double mag = pow(w * p[2], al);
          double sn, cs;
          sincos(al * PI / 2, &sn, &cs);
          const cplx den = c_pow(cplx{1.0 + mag * cs, mag * sn}, be);
          const double dd = den.re * den.re + den.im * den.im;
          e = {p[0] + p[1] * den.re / dd, -p[1] * den.im / dd};
          break;
        }
        case DEBYE_MODEL_JONSCHER: {
          const double f = p[1] * pow(w / p[2], p[3] - 1.0);
          e = {p[0] + f, -f / tan(p[3] * PI / 2)};
          break;
        }
        case DEBYE_MODEL_JONSCHER_EQ5: {
          const double f = p[1] * pow(w / p[2], p[3]);
          double sn, cs;
          sincos(p[3] * PI / 2, &sn, &cs);
          e = {p[0] + f * cs, -f * sn};
          break;
        }
        case DEBYE_MODEL_CRIM: {
          const double a = p[0];
          const int nc = (int)p[1];
          cplx acc = {0.0, 0.0};
          for (int i = 0; i < nc && i < 3; ++i)
            acc = c_add(acc, c_scale(c_pow(c_debye(p[5 + 3 * i], p[6 + 3 * i], w * p[7 + 3 * i]), a), p[2 + i]));
          e = c_pow(acc, 1.0 / a);
          break;
        }
        case DEBYE_MODEL_DEBYE_SUM: {
          e = {p[0], 0.0};
          for (int64_t j = pole_off[s]; j < pole_off[s + 1]; ++j) e = c_add(e, c_debye(0.0, pdeps[j], w * ptau[j]));
          const double f = p[1] * pow(w / p[2], p[3] - 1.0);
          e = c_add(e, cplx{f, -f / tan(p[3] * PI / 2)});
          sigma = p[4];
          break;
        }
        default:
          set_status(status, DEBYE_EBOUNDS);
      }
      double vr = e.re, vi = -e.im;   // eps' and eps'' (Eq. 1)
      if (nre && sigma != 0.0) {
        vr *= 1.0 + sigma * nre[k];
        vi *= 1.0 + sigma * nim[k];
      }
      er[k] = vr;
      ei[k] = vi;
    }
  }
}

void launch_synth(int64_t S, const int64_t* offsets, const double* omega, const int32_t* model,
                  const double* params, const int64_t* pole_off, const double* ptau,
                  const double* pdeps, const double* nre, const double* nim, double* er, double* ei,
                  int* status, int sms, cudaStream_t st) {
  if (S <= 0) return;
  int grid = (int)std::min<int64_t>(S, (int64_t)sms * 8);
  k_synth<<<grid, 256, 0, st>>>(S, offsets, omega, model, params, pole_off, ptau, pdeps, nre, nim,
                                er, ei, status);
}

}  // namespace debyefit
