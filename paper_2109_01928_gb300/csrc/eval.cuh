// Per-N passes over the frequency samples of one candidate.
//
// Thread mapping: a group of `ks` consecutive lanes (ks = a.ks, a power of two
// <= 32) evaluates one candidate; lane `slice` of the group sums the samples
// k0 + slice, k0 + slice + ks, ... and the group then reduces its partial sums
// with warp shuffles. All lanes of a block belong to the same spectrum. ks = 1
// (one thread per candidate, every per-sample load a warp-wide broadcast) is
// used for full populations; ks > 1 keeps warps full when a spectrum has only
// a few candidates (line-search points, one re-solve per spectrum).
//
// Mixed precision (float-float on the FP32 pipe):
//   sums_sq_unit column sums S_i = sum re_i and h = A^T b of the Debye basis (and,
//                for the gradient, the same sums over the derivative columns),
//                from which the column-sum solve forms the Gram, weights, cost and gradient.
// FP64 precision:
//   gram_unit    G = A^T A (packed, (N+1)x(N+1)) and h = A^T b of the stacked
//                real basis of Eq. 7 (rows: eps' and eps'' of every sample).
//   refine_unit  r = b - A x at the current weights, rr = ||r||^2 and t = A^T r.
//   grad_unit    projections of the derivative columns needed by the
//                variable-projection gradient.
//
// No lane returns before the group reduction: lanes without a candidate (the
// tail of a unit, masked line-search points) contribute zeros.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "solve_warp.cuh"

namespace debyefit {

template <int N>
struct Acc {
  static constexpr int NP = N * (N + 1) / 2;
};


// ------------------------------------------------------------------ group reductions
__device__ __forceinline__ float group_sum(float v, int ks) {
  for (int o = ks >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double group_sum(double v, int ks) {
  for (int o = ks >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Float-float sum over the group: leading parts by TwoSum, low parts added.
__device__ __forceinline__ void group_sum_ff(float& h, float& l, int ks) {
  for (int o = ks >> 1; o > 0; o >>= 1) {
    const float h2 = __shfl_xor_sync(0xffffffffu, h, o);
    const float l2 = __shfl_xor_sync(0xffffffffu, l, o);
    float s, e;
    two_sum(h, h2, s, e);
    h = s;
    l = __fadd_rn(__fadd_rn(l, l2), e);
  }
}

struct Lane {
  int q;       // candidate
  int slice;   // sample phase within the group
  int ks;      // lanes per candidate
  bool act;    // this lane's candidate is evaluated
};

__device__ __forceinline__ Lane lane_of(const EvalArgs& a, const Unit& u, bool need_ok) {
  Lane l;
  l.ks = a.ks;
  l.slice = (int)threadIdx.x & (a.ks - 1);
  l.q = u.q0 + (int)threadIdx.x / a.ks;
  l.act = l.q < u.q1;
  if (l.act && a.active) l.act = a.active[l.q] != 0;
  if (l.act && need_ok) l.act = a.sc.fail[l.q] == 0;
  return l;
}

// ------------------------------------------------------------------ Gram
template <int N>
__device__ __forceinline__ void gram_unit(const EvalArgs& a, const Unit& u) {
  const Lane ln = lane_of(a, u, false);
  const int q = ln.act ? ln.q : u.q0;
  constexpr int NP = Acc<N>::NP;
  const double* th = a.theta + (int64_t)q * a.sc.nmax;
  const int64_t Q = a.sc.Q;
  const int64_t kbeg = u.k0 + ln.slice;
  double tau[N], g0[N], hv[N], gp[NP];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    tau[i] = ln.act ? exp10(th[i]) : 0.0;
    g0[i] = 0.0;
    hv[i] = 0.0;
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) gp[i] = 0.0;
  const int64_t kend = ln.act ? u.k1 : kbeg;
#pragma unroll 1
  for (int64_t k = kbeg; k < kend; k += ln.ks) {
    const double w = __ldg(&a.omega[k]);
    const double br = __ldg(&a.eps_re[k]);
    const double bi = __ldg(&a.eps_im[k]);
    double re[N], im[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const double x = w * tau[i];
      const double r = rcp_ge1(fma(x, x, 1.0));
      re[i] = r;
      im[i] = x * r;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      g0[i] += re[i];
      hv[i] = fma(re[i], br, fma(im[i], bi, hv[i]));
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int j = 0; j <= i; ++j)
        gp[i * (i + 1) / 2 + j] = fma(re[i], re[j], fma(im[i], im[j], gp[i * (i + 1) / 2 + j]));
  }
  const bool wr = ln.act && ln.slice == 0;
  double* G = a.sc.G;
  const int hb = (a.sc.nmax + 1) * (a.sc.nmax + 2) / 2;
  if (wr) {
    G[(int64_t)pk(0, 0) * Q + q] = (double)(u.k1 - u.k0);
    G[(int64_t)hb * Q + q] = a.h0[u.s];
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const double g0s = group_sum(g0[i], ln.ks);
    const double hs = group_sum(hv[i], ln.ks);
    if (wr) {
      G[(int64_t)pk(i + 1, 0) * Q + q] = g0s;
      G[(int64_t)(hb + 1 + i) * Q + q] = hs;
    }
#pragma unroll
    for (int j = 0; j <= i; ++j) {
      const double v = group_sum(gp[i * (i + 1) / 2 + j], ln.ks);
      if (wr) G[(int64_t)pk(i + 1, j + 1) * Q + q] = v;
    }
  }

}

// ------------------------------------------------------------------ Gram from FP64 column sums
// The FP64 path's Gram G and h = A^T b by the partial-fraction identity of the Debye
// columns (the mixed path's algebra, in plain FP64): the pass sums, per pole,
//   S_i = sum_k re_i(k),   h_i = sum_k re_i(k) eps'_k + tau_i sum_k re_i(k) (omega_k eps''_k)
// (im = omega tau re) with re = 1/(1 + omega^2 tau^2), and writes the packed Gram
//   G_00 = K, G_i0 = G_ii = S_i, G_ij = (tau_i S_i + tau_j S_j) / (tau_i + tau_j)
// in gram_unit's layout, so the FP64 solve, residual passes and finish follow unchanged
// (the cost comes from the residual pass, free of the cancellation of b^T b - x^T h).
template <int N>
__device__ __forceinline__ void gram_sums_unit(const EvalArgs& a, const Unit& u) {
  const Lane ln = lane_of(a, u, false);
  const int q = ln.act ? ln.q : u.q0;
  const double* th = a.theta + (int64_t)q * a.sc.nmax;
  const int64_t Q = a.sc.Q;
  const int64_t kbeg = u.k0 + ln.slice;
  const int64_t kend = ln.act ? u.k1 : kbeg;
  double tau[N], t2[N], sv[N], av[N], bv[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    tau[i] = ln.act ? exp10(th[i]) : 0.0;
    t2[i] = tau[i] * tau[i];
    sv[i] = av[i] = bv[i] = 0.0;
  }
#pragma unroll 1
  for (int64_t k = kbeg; k < kend; k += ln.ks) {
    const double w = __ldg(&a.omega[k]);
    const double er = __ldg(&a.eps_re[k]);
    const double wei = w * __ldg(&a.eps_im[k]);
    const double w2 = w * w;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const double r = rcp_ge1(fma(w2, t2[i], 1.0));
      sv[i] += r;
      av[i] = fma(r, er, av[i]);
      bv[i] = fma(r, wei, bv[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    sv[i] = group_sum(sv[i], ln.ks);
    av[i] = group_sum(av[i], ln.ks);
    bv[i] = group_sum(bv[i], ln.ks);
  }
  if (!(ln.act && ln.slice == 0)) return;
  double* G = a.sc.G;
  const int hb = (a.sc.nmax + 1) * (a.sc.nmax + 2) / 2;
  G[(int64_t)pk(0, 0) * Q + q] = (double)(u.k1 - u.k0);
  G[(int64_t)hb * Q + q] = a.h0[u.s];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    G[(int64_t)pk(i + 1, 0) * Q + q] = sv[i];
    G[(int64_t)pk(i + 1, i + 1) * Q + q] = sv[i];
    G[(int64_t)(hb + 1 + i) * Q + q] = av[i] + tau[i] * bv[i];
#pragma unroll
    for (int j = 0; j < i; ++j)
      G[(int64_t)pk(i + 1, j + 1) * Q + q] = (tau[i] * sv[i] + tau[j] * sv[j]) / (tau[i] + tau[j]);
  }
}

// ------------------------------------------------------------------ residual pass
// Reads the weights x (FP64) of candidate q, writes rt[0] = ||b - A x||^2 and
// rt[1 + j] = (A^T (b - A x))_j, j = 0..N.
template <int N>
__device__ __forceinline__ void refine_unit(const EvalArgs& a, const Unit& u) {
  const Lane ln = lane_of(a, u, true);
  const int q = ln.act ? ln.q : u.q0;
  const double* th = a.theta + (int64_t)q * a.sc.nmax;
  const int64_t Q = a.sc.Q;
  const double* X = a.sc.x;
  const int64_t kbeg = u.k0 + ln.slice;
  const int64_t kend = ln.act ? u.k1 : kbeg;
  const int64_t step = ln.ks;
  double tau[N], w[N], t[N];
  const double w0 = ln.act ? X[q] : 0.0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    tau[i] = ln.act ? exp10(th[i]) : 0.0;
    w[i] = ln.act ? X[(int64_t)(i + 1) * Q + q] : 0.0;
    t[i] = 0.0;
  }
  double t0 = 0.0, rr = 0.0;
#pragma unroll 1
  for (int64_t k = kbeg; k < kend; k += step) {
    const double om = __ldg(&a.omega[k]);
    double ar = __ldg(&a.eps_re[k]) - w0;
    double ai = __ldg(&a.eps_im[k]);
    double re[N], im[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const double x = om * tau[i];
      const double r = rcp_ge1(fma(x, x, 1.0));
      re[i] = r;
      im[i] = x * r;
      ar = fma(-w[i], re[i], ar);
      ai = fma(-w[i], im[i], ai);
    }
    rr = fma(ar, ar, fma(ai, ai, rr));
    t0 += ar;
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = fma(re[i], ar, fma(im[i], ai, t[i]));
  }
  rr = group_sum(rr, ln.ks);
  t0 = group_sum(t0, ln.ks);
#pragma unroll
  for (int i = 0; i < N; ++i) t[i] = group_sum(t[i], ln.ks);
  if (ln.act && ln.slice == 0) {
    double* R = a.sc.rt;
    R[q] = rr;
    R[Q + q] = t0;
#pragma unroll
    for (int i = 0; i < N; ++i) R[(int64_t)(i + 2) * Q + q] = t[i];
  }

}

// ------------------------------------------------------------------ sample staging (bulk copies)
// The column-sum pass reads, for every sample of a unit's spectrum, one float4 of each
// of the three sample planes of EvalArgs; every lane of the block reads the same samples.
// They are staged in shared memory in chunks of STAGE_SAMPLES by the Tensor Memory
// Accelerator (cp.async.bulk, a plain global -> shared copy completing on an mbarrier),
// double-buffered: thread 0 issues chunk c + 1 while the block computes on chunk c. Every
// record is 16 bytes and 16-byte aligned, as the bulk copy requires. The chunk is a
// multiple of the most lanes per candidate (32), so that a lane's samples keep their
// stride across chunks; 37 KB per block leave room for 6 blocks per SM. (Chunks of 128,
// with twice the blocks' room but three times the barriers: 1024 spectra x 8 candidates,
// 8 lanes each, with the gradient 383 us against 357 us; 256 candidates, one lane each,
// 1626 against 1597 us.)
//
// Every wait on an mbarrier is bounded (STAGE_WAIT_CYCLES of clock64): a wait that
// runs out records DEBYE_ETIMEOUT, the block agrees on it (__syncthreads_or), waits
// again, bounded, for its own copies still in flight, and leaves the kernel.
constexpr int STAGE_SAMPLES = 384;
constexpr int STAGE_GRANULES = STAGE_SAMPLES / GRANULE;
static_assert(STAGE_SAMPLES % GRANULE == 0 && STAGE_SAMPLES % 32 == 0, "a chunk is whole granules and whole lane groups");
constexpr int STAGE_BUF = 3 * STAGE_SAMPLES + STAGE_GRANULES;   // float4 records of one buffer
constexpr int STAGE_RECORDS = 2 * STAGE_BUF;
constexpr long long STAGE_WAIT_CYCLES = 1ll << 31;   // about 1 s at the maximum SM clock

struct Stage {
  float4* buf;       // [2][3 planes of STAGE_SAMPLES, then STAGE_GRANULES]
  uint64_t* bar;     // [2] one mbarrier per buffer
  uint32_t fills0, fills1;     // completed phases of each buffer (the same in every thread)
  bool pending0, pending1;     // a copy into the buffer has been issued and not yet waited for
  __device__ __forceinline__ uint32_t& fills(int b) { return b ? fills1 : fills0; }
  __device__ __forceinline__ bool& pending(int b) { return b ? pending1 : pending0; }
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void stage_init(Stage& st, float4* buf, uint64_t* bar) {
  st.buf = buf;
  st.bar = bar;
  st.fills0 = st.fills1 = 0;
  st.pending0 = st.pending1 = false;
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar + b)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

// Thread 0: copy samples k .. k + n - 1 of the three planes, and their granules (from g),
// into buffer b.
__device__ __forceinline__ void stage_issue(const EvalArgs& a, Stage& st, int b, int64_t k, int64_t g, int n) {
  if (threadIdx.x == 0) {
    const uint32_t bytes = (uint32_t)n * (uint32_t)sizeof(float4);
    const uint32_t gbytes = (uint32_t)((n + GRANULE - 1) / GRANULE) * (uint32_t)sizeof(float4);
    const uint32_t bar = smem_addr(st.bar + b);
    float4* dst = st.buf + b * STAGE_BUF;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // earlier generic reads of the buffer
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(3u * bytes + gbytes) : "memory");
    const float4* src[4] = {a.kq0 + k, a.kq1 + k, a.kq2 + k, a.kg + g};
#pragma unroll
    for (int p = 0; p < 4; ++p)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(smem_addr(dst + p * STAGE_SAMPLES)), "l"(src[p]), "r"(p < 3 ? bytes : gbytes), "r"(bar) : "memory");
  }
  st.pending(b) = true;
}

// Wait (bounded) until buffer b's current phase has completed.
__device__ __forceinline__ bool stage_wait_one(Stage& st, int b) {
  const uint32_t bar = smem_addr(st.bar + b), parity = st.fills(b) & 1u;
  const long long t0 = clock64();
  uint32_t done = 0;
  while (true) {
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    if (done || clock64() - t0 > STAGE_WAIT_CYCLES) break;
  }
  if (done) {
    st.fills(b) += 1;
    st.pending(b) = false;
  }
  return done != 0;
}

// Buffer b ready in every thread; false (the block agreeing) if a wait ran out.
__device__ __forceinline__ bool stage_wait(const EvalArgs& a, Stage& st, int b) {
  const bool ok = stage_wait_one(st, b);
  if (__syncthreads_or(!ok)) {
    if (threadIdx.x == 0) set_status(a.status, DEBYE_ETIMEOUT);
    for (int c = 0; c < 2; ++c)
      if (st.pending(c)) stage_wait_one(st, c);   // the block's own copies in flight
    return false;
  }
  return true;
}

// ------------------------------------------------------------------ column-sum pass (mixed)
// For the mixed evaluation from column sums (solve_sums.cuh): per candidate, in
// float-float,
//   S_i = sum_k re_i(k)                      (the pole block of the Gram follows from these)
//   h_i = sum_k re_i(k) eps'_k + im_i(k) eps''_k   (A^T b without the eps_inf row)
// and, with the gradient (GRAD), the same sums over the derivative columns
// d/d theta_i (theta = log10 tau):
//   D_i = sum_k d re_i(k),   E_i = sum_k d re_i(k) eps'_k + d im_i(k) eps''_k.
// The basis needs only x^2 = omega^2 tau^2: one float-float product of the
// per-sample omega^2 and the per-candidate tau^2 (scaled by 2^-60 and 2^60,
// exactly, to keep both far from the float range limits); 1 + x^2 by Fast2Sum on
// (max, min); re = 1/(1 + x^2) by the approximate reciprocal and one Newton step.
// With im = x re = omega tau re,
//   h_i = sum_k re_i(k) eps'_k + tau_i B_i,   B_i = sum_k re_i(k) (omega_k eps''_k),
// two Dot2 sums on the per-sample eps' and omega eps'' (k_prep_samples stores
// omega^2, eps' and omega eps'' in a.kq0, a.kq1, a.kq2). With u = x^2 re^2 = re (1 - re),
// d re / d theta = -2 ln10 u and d im / d theta = ln10 x re^2 (1 - x^2)
// = ln10 omega tau (re - 2u), so
//   D_i = -2 ln10 U_i,   E_i = ln10 (-2 V_i + tau_i (B_i - 2 W_i)),
//   U = sum u,  V = sum u eps',  W = sum u (omega eps'').
// The same-sign sums S (re <= 1) and U (u <= 1/4) start from a bias of 1 so that
// Fast2Sum is exact; the bias is removed at the end. Writes tau_i = 10^theta_i to
// sc.x[i Q + q] (the FP64 power is done once per candidate here rather than again
// in the solve), sc.G[i Q + q] = S_i, sc.G[(N + i) Q + q] = h_i, and with GRAD
// sc.G[(2N + i) Q + q] = D_i, sc.G[(3N + i) Q + q] = E_i: in float-float, as the solves
// read them.
//
// The steps of one pole (V = float) or of a pair of poles (V = float2).
template <class V, bool GRAD>
struct SumAcc {
  V t2h, t2l;                       // (tau 2^30)^2
  V sh, sl, ah, al, ch, cl;         // S + 1, sum re eps', sum re omega eps''
  V uh, ul, vh, vl, wh, wl;         // GRAD: U + 1, V, W
};

// One sample of the three planes, every part twice.
struct SamplePair {
  float2 w2h, w2l, erh, erl, cih, cil;
  __device__ __forceinline__ void load(const float4* p) {
    const float4 a = p[0], b = p[STAGE_SAMPLES], c = p[2 * STAGE_SAMPLES];
    w2h = make_float2(a.x, a.y);
    w2l = make_float2(a.z, a.w);
    erh = make_float2(b.x, b.y);
    erl = make_float2(b.z, b.w);
    cih = make_float2(c.x, c.y);
    cil = make_float2(c.z, c.w);
  }
};

template <bool ORDERED, class V, bool GRAD>
__device__ __forceinline__ void sums_sq_step(SumAcc<V, GRAD>& t, const SamplePair& smp) {
  V w2h, w2l, erh, erl, cih, cil;
  v_part(smp.w2h, w2h);
  v_part(smp.w2l, w2l);
  v_part(smp.erh, erh);
  v_part(smp.erl, erl);
  v_part(smp.cih, cih);
  v_part(smp.cil, cil);
  // x^2 in float-float (the product of the low parts, ~2^-48, is dropped)
  const V x2h = v_mul(w2h, t.t2h);
  V x2l = v_fma(w2h, t.t2h, v_neg(x2h));
  x2l = v_fma(w2h, t.t2l, v_fma(w2l, t.t2h, x2l));
  // d = 1 + x^2: Fast2Sum of (max, min), exact
  V big, small;
  v_order1(x2h, big, small);
  const V dh = v_add(big, small);
  const V dl = v_add(v_sub(small, v_sub(dh, big)), x2l);
  // re = 1/d: approximate reciprocal and one Newton step on the float-float d
  const V r0 = v_rcp(dh);
  V e = v_fma(v_neg(dh), r0, v_all<V>(1.0f));
  e = v_fma(v_neg(dl), r0, e);
  const V rl = v_mul(r0, e);
  v_add_pos(t.sh, t.sl, r0, rl);                         // sh >= 1 >= re
  v_add_prod<ORDERED>(t.ah, t.al, r0, rl, erh, erl);              // re eps'
  v_add_prod<ORDERED>(t.ch, t.cl, r0, rl, cih, cil);              // re omega eps''
  if constexpr (GRAD) {
    V r2h, r2l, qh, ql;
    v_mul_ff(r0, rl, r0, rl, r2h, r2l);                  // re^2
    v_mul_ff(x2h, x2l, r2h, r2l, qh, ql);                // u = x^2 re^2
    v_add_pos(t.uh, t.ul, qh, ql);                       // uh >= 1 >= u
    v_add_prod<ORDERED>(t.vh, t.vl, qh, ql, erh, erl);            // u eps'
    v_add_prod<ORDERED>(t.wh, t.wl, qh, ql, cih, cil);            // u omega eps''
  }
}

__device__ __forceinline__ float& v_half(float2& v, int k) { return k ? v.y : v.x; }
__device__ __forceinline__ float& v_half(float& v, int) { return v; }

// tau = 10^theta of pole j and the float-float (tau 2^30)^2. One call site per kernel
// serves every pole: the FP64 power is about 25 FP64 instructions, each of which holds a
// sub-partition's FP64 pipe for 64 cycles on this GPU.
static __device__ __noinline__ double sums_tau(double theta, float& h, float& l) {
  const double tau = exp10(theta);
  const double ts = tau * 0x1p30;
  const ff t2 = ff_of(ts * ts);
  h = t2.h;
  l = t2.l;
  return tau;
}

template <class V, bool GRAD>
__device__ __forceinline__ void sums_sq_zero(SumAcc<V, GRAD>& t, int k) {
  v_half(t.sh, k) = 1.f;
  v_half(t.sl, k) = v_half(t.ah, k) = v_half(t.al, k) = v_half(t.ch, k) = v_half(t.cl, k) = 0.f;
  if constexpr (GRAD) {
    v_half(t.uh, k) = 1.f;
    v_half(t.ul, k) = v_half(t.vh, k) = v_half(t.vl, k) = v_half(t.wh, k) = v_half(t.wl, k) = 0.f;
  }
}

// The group's totals of one pole.
template <bool GRAD>
struct PoleSums {
  float sh, sl, ah, al, ch, cl, uh, ul, vh, vl, wh, wl;
  template <class V>
  __device__ __forceinline__ void reduce(SumAcc<V, GRAD>& t, int k, int ks) {
    sh = v_half(t.sh, k), sl = v_half(t.sl, k), ah = v_half(t.ah, k), al = v_half(t.al, k);
    ch = v_half(t.ch, k), cl = v_half(t.cl, k);
    group_sum_ff(sh, sl, ks);
    group_sum_ff(ah, al, ks);
    group_sum_ff(ch, cl, ks);
    if constexpr (GRAD) {
      uh = v_half(t.uh, k), ul = v_half(t.ul, k), vh = v_half(t.vh, k), vl = v_half(t.vl, k);
      wh = v_half(t.wh, k), wl = v_half(t.wl, k);
      group_sum_ff(uh, ul, ks);
      group_sum_ff(vh, vl, ks);
      group_sum_ff(wh, wl, ks);
    }
  }
};

// S, h (and D, E) of one pole in FP64, stored in float-float with tau (or as they are:
// sums_f64): tau at x[0], the sums at G[0], G[dn], G[2 dn], G[3 dn]. One copy of the code
// per kernel, called for every pole.
template <bool GRAD>
static __device__ __noinline__ void sums_write(double* x, double* G, int64_t dn, PoleSums<GRAD> s, int ks,
                                               bool sums_f64) {
  constexpr double LN10 = 2.302585092994046;
  const double tau = x[0];
  const double B = dbl_of(s.ch) + dbl_of(s.cl);
  const double h = (dbl_of(s.ah) + dbl_of(s.al)) + tau * B;
  // The bias is removed exactly. A lane's sh, grown by terms of at most 1, stays at most 2^24
  // (2^24 + 1 is a tie that rounds to 2^24; what is lost goes to sl), so the ks lanes' total is
  // at most ks 2^24: its last bit is at most ks, a power of two, and sh - ks a multiple of it
  // that needs no more bits than sh. The same holds for uh. The sum's FP64 rounding is then that
  // of its low part.
  ff S;
  two_sum(__fsub_rn(s.sh, (float)ks), s.sl, S.h, S.l);
  double D = 0.0, E = 0.0;
  if constexpr (GRAD) {
    const double U = dbl_of(__fsub_rn(s.uh, (float)ks)) + dbl_of(s.ul);
    const double Vs = dbl_of(s.vh) + dbl_of(s.vl);
    const double W = dbl_of(s.wh) + dbl_of(s.wl);
    D = -2.0 * LN10 * U;
    E = LN10 * (-2.0 * Vs + tau * (B - 2.0 * W));
  }
  if (sums_f64) {
    G[0] = dbl_of(S.h) + dbl_of(S.l);
    G[dn] = h;
    if constexpr (GRAD) {
      G[2 * dn] = D;
      G[3 * dn] = E;
    }
  } else {
    store_ff(x, 0, ff_of(tau));
    store_ff(G, 0, ff_round53(S));
    store_ff(G, dn, ff_of(h));
    if constexpr (GRAD) {
      store_ff(G, 2 * dn, ff_of(D));
      store_ff(G, 3 * dn, ff_of(E));
    }
  }
}

// Every product that a granule adds to the sums of half k of t is at most the accumulator
// it is added to: re <= 1 / (1 + w2min tau^2) and u = re (1 - re) <= min(re, 1/4, x^2) up
// to rounding (2^-21, covered by the factor), and the accumulators only grow while the
// granule's values are >= 0. The granule's infinite bounds compare false.
template <class V, bool GRAD>
__device__ __forceinline__ bool sums_sq_ordered(SumAcc<V, GRAD>& t, int k, float4 g) {
  const float t2 = v_half(t.t2h, k);
  const float re = rcp_approx(__fmaf_rn(g.x, t2, 1.f)) * 1.00001f;
  bool ok = v_half(t.ah, k) >= g.y * re && v_half(t.ch, k) >= g.z * re;
  if constexpr (GRAD) {
    const float u = fminf(fminf(re, 0.25f), g.w * t2) * 1.00001f;
    ok = ok && v_half(t.vh, k) >= g.y * u && v_half(t.wh, k) >= g.z * u;
  }
  return ok;
}

// One sweep over the samples for poles P0 .. P0 + C - 1 of an N-pole candidate, two poles
// per packed step (an odd last pole takes the scalar step). The FP64 work per pole (tau,
// and the final sums) is dealt out to the group's lanes, pole i to lane i mod ks.
//
// What bounds it: operand reads from the register file. A packed addition reads 4
// registers and a packed FMA 6 of the 2 that a sub-partition delivers per cycle (measured
// 2.0 and 3.0 cycles per warp instruction), so the 40 operations of a (sample, pole)
// cannot run at the FP32 pipe's 40 cycles; scalar instructions cost the same reads at
// twice the issue slots (62 cycles per (sample, pole) for N = 12 before, 57 packed). What
// is left is to issue fewer of them: where a granule's bounds show that no product can
// exceed the accumulator it is added to, the exact sum needs 3 additions instead of 6,
// with the same error term. 47 cycles now: N = 12, 128 spectra x 512 candidates x 1024
// samples at 64 candidates x 2 lanes 1.259 -> 0.941 ms, N = 20 2.512 -> 1.558 ms, N = 2
// 0.233 -> 0.184 ms; derivative sums N = 8 1.474 -> 1.158 ms. Every rounding is unchanged.
template <int N, int P0, int C, bool GRAD>
__device__ __forceinline__ bool sums_sq_sweep(const EvalArgs& a, const Unit& u, const Lane& ln, int q, Stage& st) {
  constexpr int CP = C / 2, ODD = C & 1;
  constexpr unsigned FULL = 0xffffffffu;
  SumAcc<float2, GRAD> pr[CP > 0 ? CP : 1];
  SumAcc<float, GRAD> odd;
  float mh = 0.f, ml = 0.f;
#pragma unroll
  for (int i = 0; i < C; ++i) {
    const int own = i & (ln.ks - 1);
    if (own == 0) {
      const int j = P0 + i + ln.slice;
      mh = ml = 0.f;
      if (ln.act && i + ln.slice < C) a.sc.x[(int64_t)j * a.sc.Q + q] = sums_tau(a.theta[(int64_t)q * a.sc.nmax + j], mh, ml);
    }
    const float h = __shfl_sync(FULL, mh, own, ln.ks), l = __shfl_sync(FULL, ml, own, ln.ks);
    if (i < 2 * CP) {
      v_half(pr[i / 2].t2h, i & 1) = h;
      v_half(pr[i / 2].t2l, i & 1) = l;
      sums_sq_zero(pr[i / 2], i & 1);
    } else {
      odd.t2h = h;
      odd.t2l = l;
      sums_sq_zero(odd, 0);
    }
  }
  const int64_t nk = u.k1 - u.k0, g0 = granule_base(u.k0, u.s);
  const int nch = (int)((nk + STAGE_SAMPLES - 1) / STAGE_SAMPLES);
  auto chunk_len = [&](int64_t c0) { return (int)(nk - c0 < STAGE_SAMPLES ? nk - c0 : STAGE_SAMPLES); };
  // Samples per check of the order: 16 of every lane; from 8 lanes on the whole chunk (a
  // check per 128 samples costs more than the ordered sums gain there: 1024 spectra x 8
  // candidates with the gradient 369 us against 357 us)
  const int run = ln.ks <= 2 ? GRANULE : ln.ks <= 4 ? 2 * GRANULE : STAGE_SAMPLES;
  if (nch > 0) stage_issue(a, st, 0, u.k0, g0, chunk_len(0));
#pragma unroll 1
  for (int c = 0; c < nch; ++c) {
    const int b = c & 1;
    const int64_t c0 = (int64_t)c * STAGE_SAMPLES;
    if (c + 1 < nch)   // buffer b ^ 1 was released by the barrier that ended chunk c - 1
      stage_issue(a, st, b ^ 1, u.k0 + c0 + STAGE_SAMPLES, g0 + (int64_t)(c + 1) * STAGE_GRANULES,
                  chunk_len(c0 + STAGE_SAMPLES));
    if (!stage_wait(a, st, b)) return false;
    const float4* buf = st.buf + b * STAGE_BUF;
    const int cnt = chunk_len(c0);
#pragma unroll 1
    for (int jb = 0; jb < cnt; jb += run) {
      const int je = jb + run < cnt ? jb + run : cnt;
      float4 g = buf[3 * STAGE_SAMPLES + jb / GRANULE];
      for (int gi = jb + GRANULE; gi < je; gi += GRANULE) {
        const float4 h = buf[3 * STAGE_SAMPLES + gi / GRANULE];
        g = make_float4(fminf(g.x, h.x), fmaxf(g.y, h.y), fmaxf(g.z, h.z), fmaxf(g.w, h.w));
      }
      bool fast = true;
#pragma unroll
      for (int i = 0; i < CP; ++i) fast = fast && sums_sq_ordered(pr[i], 0, g) && sums_sq_ordered(pr[i], 1, g);
      if constexpr (ODD) fast = fast && sums_sq_ordered(odd, 0, g);
      const int jend = ln.act ? je : 0;
      auto sweep = [&](auto ordered) {
        constexpr bool ORD = decltype(ordered)::value;
        constexpr int U = 2;   // samples per step: their reciprocals and products overlap
        int j = jb + ln.slice;
        auto one = [&](const SamplePair& smp) {
#pragma unroll
          for (int i = 0; i < CP; ++i) sums_sq_step<ORD>(pr[i], smp);
          if constexpr (ODD) sums_sq_step<ORD>(odd, smp);
        };
#pragma unroll 1
        for (; j + (U - 1) * ln.ks < jend; j += U * ln.ks) {
          SamplePair smp[U];
#pragma unroll
          for (int v = 0; v < U; ++v) smp[v].load(buf + j + v * ln.ks);
#pragma unroll
          for (int v = 0; v < U; ++v) one(smp[v]);
        }
#pragma unroll 1
        for (; j < jend; j += ln.ks) {
          SamplePair smp;
          smp.load(buf + j);
          one(smp);
        }
      };
      if (__all_sync(FULL, fast || !ln.act)) sweep(std::true_type{});
      else sweep(std::false_type{});
    }
    __syncthreads();   // the whole block is done with buffer b
  }
  PoleSums<GRAD> mine, t;
#pragma unroll
  for (int i = 0; i < C; ++i) {
    const int own = i & (ln.ks - 1);
    if (i < 2 * CP) t.reduce(pr[i / 2], i & 1, ln.ks);
    else t.reduce(odd, 0, ln.ks);
    if (own == ln.slice) mine = t;
    if (own == ln.ks - 1 || i == C - 1) {
      const int k = i - own + ln.slice;   // this lane's pole of the group's last ks poles
      if (ln.act && k < C) {
        const int64_t at = (int64_t)(P0 + k) * a.sc.Q + q;
        sums_write<GRAD>(a.sc.x + at, a.sc.G + at, N * a.sc.Q, mine, ln.ks, a.sums_f64 != 0);
      }
    }
  }
  return true;
}

// Poles P0 .. N - 1 in sweeps of at most CH poles each, an even number wherever possible.
template <int N, int P0, int CH, bool GRAD>
__device__ __forceinline__ bool sums_sq_sweeps(const EvalArgs& a, const Unit& u, const Lane& ln, int q, Stage& st) {
  constexpr int REST = N - P0, NS = (REST + CH - 1) / CH;          // sweeps still to make
  constexpr int EVEN = ((REST + NS - 1) / NS + 1) / 2 * 2;         // their size, rounded up to even
  constexpr int C = EVEN < REST ? (EVEN <= CH ? EVEN : CH) : REST;
  if (!sums_sq_sweep<N, P0, C, GRAD>(a, u, ln, q, st)) return false;
  if constexpr (P0 + C < N) return sums_sq_sweeps<N, P0 + C, CH, GRAD>(a, u, ln, q, st);
  return true;
}

// A unit without any active candidate (a masked evaluation) is skipped by the whole block.
// Returns false if a wait for staged samples ran out (the block then stops).
template <int N, bool GRAD>
__device__ __forceinline__ bool sums_sq_unit(const EvalArgs& a, const Unit& u, Stage& st) {
  const Lane ln = lane_of(a, u, false);
  if (!__syncthreads_or(ln.act)) return true;
  const int q = ln.act ? ln.q : u.q0;
  return sums_sq_sweeps<N, 0, GRAD ? SQUARED_CHUNK_GRAD : SQUARED_CHUNK, GRAD>(a, u, ln, q, st);
}

// ------------------------------------------------------------------ gradient pass
// With x1 (unflipped, sc.x), x_hat (flipped, sc.xh) and w = M^-1 S g_hat (sc.w):
//   gt[i]        = a_i'^T r_hat,  r_hat = b - A x_hat
//   gt[N + i]    = a_i^T a_i'
//   gt[2N + i]   = a_i'^T r,      r = b - A x1
//   gt[3N + i]   = a_i'^T (A w)
// where a_i' = d a_i / d log10(tau_i).
template <int N>
__device__ __forceinline__ void grad_unit(const EvalArgs& a, const Unit& u) {
  const Lane ln = lane_of(a, u, true);
  const int q = ln.act ? ln.q : u.q0;
  const double* th = a.theta + (int64_t)q * a.sc.nmax;
  const int64_t Q = a.sc.Q;
  const int64_t kbeg = u.k0 + ln.slice;
  const int64_t kend = ln.act ? u.k1 : kbeg;
  const int64_t step = ln.ks;
  constexpr double LN10 = 2.302585092994046;
  auto ld = [&](const double* p) { return ln.act ? *p : 0.0; };
  double tau[N], xh[N], e[N], w[N];
  double t_rh[N], t_aa[N], t_r[N], t_aw[N];
  const double x0 = ld(a.sc.xh + q);
  const double e0 = x0 - ld(a.sc.x + q);
  const double w0 = ld(a.sc.w + q);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    tau[i] = ln.act ? exp10(th[i]) : 0.0;
    xh[i] = ld(a.sc.xh + (int64_t)(i + 1) * Q + q);
    e[i] = xh[i] - ld(a.sc.x + (int64_t)(i + 1) * Q + q);
    w[i] = ld(a.sc.w + (int64_t)(i + 1) * Q + q);
    t_rh[i] = t_aa[i] = t_r[i] = t_aw[i] = 0.0;
  }
#pragma unroll 1
  for (int64_t k = kbeg; k < kend; k += step) {
    const double om = __ldg(&a.omega[k]);
    double rhr = __ldg(&a.eps_re[k]) - x0, rhi = __ldg(&a.eps_im[k]);
    double aer = e0, aei = 0.0, awr = w0, awi = 0.0;
    double re[N], im[N], xv[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const double x = om * tau[i];
      const double r = rcp_ge1(fma(x, x, 1.0));
      xv[i] = x;
      re[i] = r;
      im[i] = x * r;
      rhr = fma(-xh[i], re[i], rhr);
      rhi = fma(-xh[i], im[i], rhi);
      aer = fma(e[i], re[i], aer);
      aei = fma(e[i], im[i], aei);
      awr = fma(w[i], re[i], awr);
      awi = fma(w[i], im[i], awi);
    }
    const double rr = rhr + aer, ri = rhi + aei;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const double x = xv[i];
      const double re2l = re[i] * re[i] * LN10;
      const double dre = -2.0 * x * x * re2l;
      const double dim = x * (1.0 - x * x) * re2l;
      t_rh[i] = fma(dre, rhr, fma(dim, rhi, t_rh[i]));
      t_aa[i] = fma(re[i], dre, fma(im[i], dim, t_aa[i]));
      t_r[i] = fma(dre, rr, fma(dim, ri, t_r[i]));
      t_aw[i] = fma(dre, awr, fma(dim, awi, t_aw[i]));
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    t_rh[i] = group_sum(t_rh[i], ln.ks);
    t_aa[i] = group_sum(t_aa[i], ln.ks);
    t_r[i] = group_sum(t_r[i], ln.ks);
    t_aw[i] = group_sum(t_aw[i], ln.ks);
  }
  if (ln.act && ln.slice == 0) {
    double* T = a.sc.gt;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      T[(int64_t)i * Q + q] = t_rh[i];
      T[(int64_t)(N + i) * Q + q] = t_aa[i];
      T[(int64_t)(2 * N + i) * Q + q] = t_r[i];
      T[(int64_t)(3 * N + i) * Q + q] = t_aw[i];
    }
  }

}

// ------------------------------------------------------------------ N dispatch
template <int PH, int N>
__device__ __forceinline__ void run_phase(const EvalArgs& a, const Unit& u) {
  if constexpr (PH == PH_GRAM) gram_unit<N>(a, u);
  else if constexpr (PH == PH_GRAM_SUMS) gram_sums_unit<N>(a, u);
  else if constexpr (PH == PH_REFINE) refine_unit<N>(a, u);
  else grad_unit<N>(a, u);
}

template <int PH, int LO, int HI>
__device__ __forceinline__ void dispatch_n(const EvalArgs& a, const Unit& u) {
  if constexpr (LO <= HI) {
    if (u.N == LO) run_phase<PH, LO>(a, u);
    else dispatch_n<PH, LO + 1, HI>(a, u);
  }
}

// The solves of a unit's candidates by the block that summed them (fuse_solve, evaluations of
// a few units): there the launch between the pass and its solve is a good part of the whole.
// The sums are read back through global memory: the block wrote them, the barrier orders
// them.
template <int N, bool GRAD>
static __device__ __noinline__ void solve_unit(const EvalArgs& a, const Unit& u) {
  __syncthreads();
  for (int q = u.q0 + ((int)threadIdx.x >> 5); q < u.q1; q += (int)blockDim.x >> 5)
    if (!a.active || a.active[q]) warp_solve<N + 1>(a, u, q, a.out_cost, a.out_weights, GRAD ? a.out_grad : nullptr);
}

// The column-sum pass (PH_SUMS, PH_SUMSG) of pole count N: one block per unit
// (grid-stride over the unit list), the unit's samples staged by bulk copies.
template <int N, bool GRAD, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_pass_sums(const __grid_constant__ EvalArgs a) {
  __shared__ __align__(128) float4 stage_buf[STAGE_RECORDS];
  __shared__ __align__(8) uint64_t stage_bar[2];
  Stage st;
  stage_init(st, stage_buf, stage_bar);
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    if (u.N != N) {
      if (threadIdx.x == 0) set_status(a.status, DEBYE_EBOUNDS);
      continue;
    }
    if (!sums_sq_unit<N, GRAD>(a, u, st)) return;
    if (a.fuse_solve) solve_unit<N, GRAD>(a, u);
  }
}

// One block per unit (grid-stride over the unit list); LO..HI is the range of pole counts
// compiled into this kernel (the library launches one N per kernel). At most MAXT threads
// per block; MINB resident blocks of that size bound the registers per thread.
template <int PH, int LO, int HI, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_pass(EvalArgs a) {
  for (int ui = blockIdx.x; ui < a.n_units; ui += gridDim.x) {
    const Unit u = a.units[ui];
    if (u.N < LO || u.N > HI) {
      if (threadIdx.x == 0) set_status(a.status, DEBYE_EBOUNDS);
      continue;
    }
    dispatch_n<PH, LO, HI>(a, u);
  }
}

}  // namespace debyefit
