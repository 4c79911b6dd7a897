// Column-sum tables of the mixed precision's table variant (DEBYE_PREC_MIXED_TABLE).
//
// The Gram identity of Debye columns (G_ij = (tau_i S_i + tau_j S_j) / (tau_i + tau_j))
// leaves, per pole, the column sums S(theta) = sum_k re_k and h(theta) = a^T b (and
// their theta derivatives for the gradient): four functions of one variable per
// spectrum, whatever the candidate. They are tabulated once per call as piecewise
// Chebyshev interpolants over the spectrum's log10(tau) box (stored as polynomials in
// the segment's coordinate), and every candidate's sums are then read off by
// float-float Horner steps: O(TAB_NC) per pole instead of O(K).
//
// Accuracy: with s = ln tau^2, each term 1 / (1 + w_k^2 e^s) has its poles at
// Im s = +-pi, so every column sum is analytic in the strip |Im s| < pi and bounded
// there by 1 / sin(Im s) times the sum of |terms|. On a segment of TAB_W = 0.2
// decades (0.92 in s) the Chebyshev coefficients then decay by about 20 per degree
// (Bernstein-ellipse bound), and 12 coefficients reach ~1e-14 relative: measured on
// the mixed and tabulated workloads in FP64 (worst 1e-14 for S and h, 8e-14 for the
// derivatives), below the float-float node sums' own rounding (~1e-12).
#include <cmath>

#include "common.cuh"
#include "eval.cuh"
#include "launch.h"

namespace debyefit {

// Chebyshev points of the first kind, the matching discrete cosine transform, and the
// monomial coefficients of the Chebyshev polynomials (integers, exact in FP64).
struct ChebConst {
  double xm[TAB_NC];            // x_m = cos(pi (m + 1/2) / NC)
  double dct[TAB_NC][TAB_NC];   // (2 / NC) cos(pi k (m + 1/2) / NC), row 0 halved
  double mono[TAB_NC][TAB_NC];  // T_j(x) = sum_k mono[j][k] x^k
};

static const ChebConst& cheb_const() {
  static ChebConst c = [] {
    ChebConst r{};
    const double pi = 3.14159265358979323846;
    for (int m = 0; m < TAB_NC; ++m) r.xm[m] = std::cos(pi * (m + 0.5) / TAB_NC);
    for (int k = 0; k < TAB_NC; ++k)
      for (int m = 0; m < TAB_NC; ++m)
        r.dct[k][m] = (k == 0 ? 1.0 : 2.0) / TAB_NC * std::cos(pi * k * (m + 0.5) / TAB_NC);
    // T_0 = 1, T_1 = x, T_{j+1} = 2 x T_j - T_{j-1}
    r.mono[0][0] = 1.0;
    if (TAB_NC > 1) r.mono[1][1] = 1.0;
    for (int j = 1; j + 1 < TAB_NC; ++j)
      for (int k = 0; k < TAB_NC; ++k)
        r.mono[j + 1][k] = (k > 0 ? 2.0 * r.mono[j][k - 1] : 0.0) - r.mono[j - 1][k];
    return r;
  }();
  return c;
}

struct TabBuild {
  ChebConst cc;
  const int32_t* qn0;      // [S + 1] first pseudo-candidate of each spectrum
  const int32_t* nseg;     // [S]
  const int64_t* seg0;     // [S]
  int32_t* done;           // [S] units of the spectrum that have ended
  float2* coef;
};

// Node thetas, pseudo-candidate-major: spectrum s owns rows qn0[s] .. qn0[s+1]-1 of
// theta_n[.][TAB_NODE_N]; node n = g NC + m (segment g, point m) sits at slot n of the
// spectrum's rows, theta = lo + TAB_W (g + 1/2 + x_m / 2); slots past the last node
// repeat it. Zeroes the spectrum's count of ended units.
__global__ void k_tab_nodes(int64_t S, const int32_t* qn0, const int32_t* nseg, const double* lo,
                            ChebConst cc, double* theta_n, int32_t* done) {
  for (int64_t s = blockIdx.x; s < S; s += gridDim.x) {
    if (threadIdx.x == 0) done[s] = 0;
    const int64_t base = (int64_t)qn0[s] * TAB_NODE_N;
    const int slots = (qn0[s + 1] - qn0[s]) * TAB_NODE_N;
    const int nodes = nseg[s] * TAB_NC;
    const double l = lo[s];
    for (int n = threadIdx.x; n < slots; n += blockDim.x) {
      const int nn = n < nodes ? n : nodes - 1;
      const int g = nn / TAB_NC, m = nn % TAB_NC;
      theta_n[base + n] = l + TAB_W * ((double)g + 0.5 + 0.5 * cc.xm[m]);
    }
  }
}

// Coefficients of segment g and function f of spectrum s from the node sums: for node n,
// pseudo-candidate q = qn0[s] + n / TAB_NODE_N and pole i = n % TAB_NODE_N, S, h, dS, dh
// stand at G[(r TAB_NODE_N + i) Qn + q], r = 0..3, and tau at X[i Qn + q]. Other blocks wrote
// them: they are read from L2 (a sector that this SM's L1 holds may be older). Called by a
// whole block; nf: the functions tabulated, the first 3 or all.
__device__ __forceinline__ void tab_coef(const TabBuild& t, const double* G, const double* X, int64_t Qn, int64_t s,
                                         int nf) {
  const ChebConst& cc = t.cc;
  const int items = t.nseg[s] * nf;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int g = it / nf, f = it % nf;
    double v[TAB_NC];
#pragma unroll
    for (int m = 0; m < TAB_NC; ++m) {
      const int n = g * TAB_NC + m;
      const int64_t q = t.qn0[s] + n / TAB_NODE_N;
      const int i = n % TAB_NODE_N;
      v[m] = __ldcg(f == 2 ? X + (int64_t)i * Qn + q : G + (int64_t)((f < 2 ? f : f - 1) * TAB_NODE_N + i) * Qn + q);
    }
    double c[TAB_NC];
#pragma unroll
    for (int k = 0; k < TAB_NC; ++k) {
      c[k] = 0.0;
#pragma unroll
      for (int m = 0; m < TAB_NC; ++m) c[k] = fma(cc.dct[k][m], v[m], c[k]);
    }
    // monomial coefficients in x (the series' coefficients fall by ~20 a degree, the
    // Chebyshev polynomials' monomial coefficients grow by at most 1 + sqrt 2: the
    // monomial form is as well conditioned on [-1, 1]). T_j has only powers of j's parity:
    // the skipped terms' factors are zero, and with the splits on the integer pipe 72 of 258
    // FP64 operations (64 cycles per warp each) fall away without a change of the results.
    float2* out = t.coef + ((t.seg0[s] + g) * TAB_NF + f) * TAB_NC;
#pragma unroll
    for (int k = 0; k < TAB_NC; ++k) {
      double a = 0.0;
#pragma unroll
      for (int j = k; j < TAB_NC; j += 2) a = fma(cc.mono[j][k], c[j], a);
      const ff r = ff_of(a);
      out[k] = make_float2(r.h, r.l);
    }
  }
}

// Node sums and coefficients: a block per unit (TAB_CB pseudo-candidates of one spectrum), and
// the block that ends a spectrum's last unit forms its coefficients. Those are bound by the
// FP64 pipe, which the sums leave idle: as a kernel of their own they took 65 us after the
// sums' 342 (1024 spectra, 40 segments, cost only); the whole evaluation of 256 candidates
// each 678 -> 648 us.
template <bool GRAD>
__global__ void __launch_bounds__(MAX_BLOCK, GRAD ? 2 : 3) k_tab_build(const __grid_constant__ EvalArgs a,
                                                                      const __grid_constant__ TabBuild t) {
  __shared__ __align__(128) float4 stage_buf[STAGE_RECORDS];
  __shared__ __align__(8) uint64_t stage_bar[2];
  __shared__ int last;
  Stage st;
  stage_init(st, stage_buf, stage_bar);
  const Unit u = a.units[blockIdx.x];
  if (!sums_sq_unit<TAB_NODE_N, GRAD>(a, u, st)) return;
  __threadfence();   // this thread's sums before the block's count
  __syncthreads();
  if (threadIdx.x == 0) {
    const int units = (t.qn0[u.s + 1] - t.qn0[u.s] + TAB_CB - 1) / TAB_CB;
    last = atomicAdd(&t.done[u.s], 1) == units - 1;
    __threadfence();
  }
  __syncthreads();
  if (last) tab_coef(t, a.sc.G, a.sc.x, a.sc.Q, u.s, GRAD ? TAB_NF : 3);
}

// f(x) = sum_k a_k x^k for x in [-1, 1] by Horner's rule in float-float. The
// coefficients (hi, lo) are read two at a time (16-byte loads: every function's TAB_NC
// coefficients start on a multiple of TAB_NC * 8 = 96 bytes).
static_assert(TAB_NC % 2 == 0 && (TAB_NC * sizeof(float2)) % 16 == 0, "paired coefficient loads");
constexpr int TAB_F4 = TAB_NC / 2;   // float4 of one function
__device__ __forceinline__ ff poly_ff(const float4* a4, ff x) {
  float4 c[TAB_F4];
#pragma unroll
  for (int i = 0; i < TAB_F4; ++i) c[i] = a4[i];
  ff acc{c[TAB_F4 - 1].z, c[TAB_F4 - 1].w};
#pragma unroll
  for (int k = TAB_NC - 2; k >= 0; --k) {
    const float4 q = c[k / 2];
    acc = ff_sum(ff_prod(acc, x), (k & 1) ? ff{q.z, q.w} : ff{q.x, q.y});
  }
  return acc;
}

// The four column sums of one pole directly over the spectrum's samples in FP64, for a
// theta outside the table (or not finite): S, h, dS/dtheta, dh/dtheta as the
// column-sum pass defines them.
template <bool GRAD>
__device__ void direct_sums(const EvalArgs& a, const Unit& u, double tau, double* out) {
  constexpr double LN10 = 2.302585092994046;
  double S = 0.0, A = 0.0, C = 0.0, U = 0.0, V = 0.0, W = 0.0;
#pragma unroll 1
  for (int64_t k = u.k0; k < u.k1; ++k) {
    const double om = a.omega[k];
    const double x = om * tau;
    const double re = 1.0 / (1.0 + x * x);
    const double er = a.eps_re[k], wi = om * a.eps_im[k];
    S += re;
    A += re * er;
    C += re * wi;
    if (GRAD) {
      const double uu = x * x * re * re;
      U += uu;
      V += uu * er;
      W += uu * wi;
    }
  }
  out[0] = S;
  out[1] = A + tau * C;
  out[2] = -2.0 * LN10 * U;
  out[3] = LN10 * (-2.0 * V + tau * (C - 2.0 * W));
}

// Segment of position uu (in segments from the table's origin), or -1 outside [0, ns]:
// the integer part from the bits of uu (the FP64 comparisons and conversions would each
// hold the FP64 pipe for 64 cycles per warp).
__device__ __forceinline__ int tab_segment(double uu, int ns) {
  const uint32_t hi = (uint32_t)__double2hiint(uu), lo = (uint32_t)__double2loint(uu);
  if (((hi << 1) | lo) == 0) return 0;   // +-0
  const int e = (int)(hi >> 20) - 1023;  // sign set: beyond every bound
  if (e < 0) return 0;
  if (e > 10) return -1;                 // 2048 and more (TAB_MAX_SEG is 1000), negative, infinite or NaN
  const uint32_t m = (hi & 0xfffffu) | 0x100000u;
  const int g = (int)(m >> (20 - e));
  if (g < ns) return g;
  return g == ns && ((m << (12 + e)) | lo) == 0 ? ns - 1 : -1;   // the upper bound itself
}

// A positive integer below 2^20 as a double.
__device__ __forceinline__ double dbl_of_int(uint32_t m) {
  const int z = __clz((int)m);
  return __hiloint2double((int)(((uint32_t)(1023 + 31 - z) << 20) + ((m << z << 1) >> 12)), 0);
}

// Column sums of every (candidate, pole) of the units from the tables, written where
// the column-sum pass writes them (tau to sc.x row i; S, h, dS, dh to G rows i, N + i,
// 2N + i, 3N + i, in float-float) for the column-sum solves. One thread per (candidate,
// pole). With the position and the results converted by integer operations, 3 FP64
// operations per pole are left of 20, whose pipe bound the kernel: 88 -> 67 us for 1024
// spectra x 256 candidates, N 2-12. After that the gathers did: a warp's poles lie in some
// 25 different segments, each a line of its own to the L1. A unit with at least two poles
// per segment of its spectrum copies the spectrum's functions to shared memory first, at an
// odd number of 16-byte words per segment, which spreads the segments over the banks:
// 67 -> 56 us. smem_seg: segments the launch has shared memory for.
template <bool GRAD>
__global__ void __launch_bounds__(128) k_tab_eval(EvalArgs a, int smem_seg) {
  constexpr int NF = GRAD ? TAB_NF : 3;           // functions read
  constexpr int GS = TAB_NF * TAB_F4, SS = NF * TAB_F4 + 1;   // float4 per segment: in memory, staged
  static_assert(SS % 2 == 1, "segments spread over the banks");
  extern __shared__ float4 tab_smem[];
  const int64_t Q = a.sc.Q;
  double* G = a.sc.G;
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    const int nc = u.q1 - u.q0, N = u.N;
    const double l = a.tab.lo[u.s];
    const int ns = a.tab.nseg[u.s];
    const float4* cs = reinterpret_cast<const float4*>(a.tab.coef) + a.tab.seg0[u.s] * GS;
    const bool staged = ns <= smem_seg && nc * N >= 2 * ns && !a.active;
    if (staged) {
      __syncthreads();   // the previous unit's functions are read
      for (int e = threadIdx.x; e < ns * (SS - 1); e += blockDim.x) {
        const int g = e / (SS - 1), c = e - g * (SS - 1);
        tab_smem[g * SS + c] = __ldg(cs + (int64_t)g * GS + c);
      }
      __syncthreads();
    }
    for (int p = threadIdx.x; p < nc * N; p += blockDim.x) {
      const int j = p / nc, q = u.q0 + p % nc;
      if (a.active && !a.active[q]) continue;
      const double th = a.theta[(int64_t)q * a.sc.nmax + j];
      const double d = th - l;
      const int g = tab_segment(d * TAB_INV_W, ns);
      ff tau, v[4];
      auto eval = [&](const float4* c, ff x) {
        v[0] = ff_round53(poly_ff(c, x));
        v[1] = ff_round53(poly_ff(c + TAB_F4, x));
        tau = ff_round53(poly_ff(c + 2 * TAB_F4, x));
        if (GRAD) {
          v[2] = ff_round53(poly_ff(c + 3 * TAB_F4, x));
          v[3] = ff_round53(poly_ff(c + 4 * TAB_F4, x));
        }
      };
      if (g >= 0) {
        // x = 2 (uu - g) - 1 in [-1, 1]
        const ff x = ff_of(fma(d, 2.0 * TAB_INV_W, -dbl_of_int(2 * g + 1)));
        if (staged) eval(tab_smem + g * SS, x);
        else eval(cs + (int64_t)g * GS, x);
      } else {
        double s[4];
        const double t = exp10(th);
        direct_sums<GRAD>(a, u, t, s);
        tau = ff_of(t);
        for (int f = 0; f < (GRAD ? 4 : 2); ++f) v[f] = ff_of(s[f]);
      }
      store_ff(a.sc.x, (int64_t)j * Q + q, tau);
      store_ff(G, (int64_t)j * Q + q, v[0]);
      store_ff(G, (int64_t)(N + j) * Q + q, v[1]);
      if (GRAD) {
        store_ff(G, (int64_t)(2 * N + j) * Q + q, v[2]);
        store_ff(G, (int64_t)(3 * N + j) * Q + q, v[3]);
      }
    }
  }
}

void launch_tab_build(const EvalArgs& a, int64_t S, const int32_t* qn0, const int32_t* nseg, const int64_t* seg0,
                      const double* lo, double* theta_n, int32_t* done, bool with_grad, float2* coef, int sms,
                      cudaStream_t st) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(S, (int64_t)sms * 32));
  k_tab_nodes<<<grid, 128, 0, st>>>(S, qn0, nseg, lo, cheb_const(), theta_n, done);
  const TabBuild t{cheb_const(), qn0, nseg, seg0, done, coef};
  if (with_grad) k_tab_build<true><<<a.n_units, TAB_CB * TAB_KS, 0, st>>>(a, t);
  else k_tab_build<false><<<a.n_units, TAB_CB * TAB_KS, 0, st>>>(a, t);
}

// max_seg: the most segments of a spectrum. Shared memory for up to 64 segments (box of 12.8
// decades, 19.5 KB, 31.7 KB with the derivatives); larger tables are read where they are.
void launch_tab_eval(const EvalArgs& a, bool grad, int max_seg, int sms, cudaStream_t st) {
  const int grid = std::max(1, std::min(a.n_units, sms * 16));
  const int seg = max_seg <= 64 ? max_seg : 0;
  const size_t smem = (size_t)seg * ((grad ? TAB_NF : 3) * TAB_F4 + 1) * sizeof(float4);
  if (grad) k_tab_eval<true><<<grid, 128, smem, st>>>(a, seg);
  else k_tab_eval<false><<<grid, 128, smem, st>>>(a, seg);
}

}  // namespace debyefit
