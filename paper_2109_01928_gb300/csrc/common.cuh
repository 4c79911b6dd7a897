// Shared device-side definitions of libdebyefit (sm_103a).
//
// Work decomposition: every evaluation works on a flat list of candidates q.
// Candidate q belongs to one spectrum; a Unit is a run of at most `cb`
// consecutive candidates of one spectrum, processed by one thread block with
// one thread per candidate. Per-candidate scratch is stored structure-of-arrays,
// element e of candidate q at base[e * Q + q], so a warp's 32 candidates touch 32
// consecutive doubles.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/debyefit.h"

namespace debyefit {

constexpr int NMAX = DEBYE_MAX_POLES;   // largest pole count
constexpr int NMAX1 = NMAX + 1;         // unknowns: eps_inf + d_eps_1..N
constexpr int NPACK_MAX = NMAX1 * (NMAX1 + 1) / 2;

// Packed lower-triangular index of (I, J), J <= I.
__host__ __device__ constexpr int pk(int I, int J) { return I * (I + 1) / 2 + J; }

enum Phase { PH_GRAM = 0, PH_REFINE = 1, PH_GRAD = 2, PH_SUMS = 3, PH_SUMSG = 4,
             // mixed precision: weights, cost (and gradient) from a bucket's column sums,
             // one thread per candidate, the pole count fixed at compile time
             PH_SOLVE = 5, PH_SOLVEG = 6,
             // FP64 column sums and the Gram from the partial-fraction identity (FP64 path)
             PH_GRAM_SUMS = 7 };
// The column-sum pass (eval.cuh) sweeps the samples for at most this many poles at a time
// (8 registers per pole, 14 with the derivative sums), two samples per step: measured on
// 128 spectra x 512 candidates x 1024 samples at 64 candidates x 2 lanes, N = 12 0.941 ms
// in sweeps of 6, 1.026 ms with one sample per step, 1.036 ms in one sweep of 12; N = 20
// 1.558 ms (8 + 6 + 6) against 1.708 ms with one sample per step. Derivative sums, N = 12:
// 1.723 ms in sweeps of 6, 1.787 ms in sweeps of 4, 1.879 ms with one sample per step.
constexpr int SQUARED_CHUNK = 8;
constexpr int SQUARED_CHUNK_GRAD = 6;

struct Unit {
  int32_t s;    // spectrum
  int32_t q0;   // first candidate
  int32_t q1;   // one past the last candidate
  int32_t N;    // poles of this spectrum
  int64_t k0;   // first sample of the spectrum
  int64_t k1;   // one past the last sample
};

// Per-call views of the candidate scratch (all device pointers).
struct Scratch {
  int64_t Q;        // candidates in this evaluation (SoA stride)
  int32_t nmax;     // pole capacity of theta / weights rows
  int32_t ng;       // per-candidate Gram record: packed (nmax+1) lower triangle + h
  double* G;        // [ng][Q]   Gram (packed) followed by h = A^T b; mixed precision: the column
                    //           sums S, h (and D, E), [N][Q] each, in float-float (float2)
  double* L;        // [npk][Q]  Cholesky factor of the scaled damped matrix
  double* dinv;     // [nmax+1][Q] 1 / sqrt(G_ii)
  double* x;        // [nmax+1][Q] current (unflipped) weights; mixed precision: tau [N][Q] in
                    //           float-float (float2)
  double* xh;       // [nmax+1][Q] flipped weights
  double* w;        // [nmax+1][Q] adjoint solve M^-1 S g_hat (gradient only)
  double* rt;       // [nmax+2][Q] rr = ||r||^2 then t = A^T r
  double* gt;       // [4*nmax][Q] gradient projections
  int32_t* fail;    // [Q] non-zero: candidate's damped matrix not positive definite
};

// Per-spectrum Chebyshev tables of the column sums (DEBYE_PREC_MIXED_TABLE). Over the
// spectrum's log10(tau) box [lo, lo + nseg TAB_W], each column sum of one Debye pole
// is a function of theta alone: S = sum_k re_k, h = a_i^T b and their theta
// derivatives (tau = 10^theta is tabulated with them). Every term 1 / (1 + w_k^2 tau^2) is analytic in the strip
// |Im ln tau^2| < pi whatever the samples, so on segments of TAB_W decades a
// Chebyshev interpolant of degree TAB_NC - 1 reaches the float-float sums' rounding.
constexpr double TAB_W = 0.2;    // decades of log10(tau) per segment
constexpr double TAB_INV_W = 5.0;   // 1 / TAB_W
constexpr int TAB_NC = 12;       // Chebyshev coefficients per segment and function
// Functions per segment: S, h and tau = 10^theta itself (an entire function, so its
// series converges faster still), which the cost needs, then dS/dtheta and dh/dtheta
// for the gradient.
constexpr int TAB_NF = 5;
// Nodes per pseudo-candidate of the table's node pass: one sweep of the column-sum pass, with
// and without the derivative sums (SQUARED_CHUNK_GRAD), so that a spectrum's nodes spread
// over as many blocks as possible. Times beside the launch (build_tables).
constexpr int TAB_NODE_N = 6;
constexpr int TAB_MAX_SEG = 1000;   // segments per spectrum (a box of at most 200 decades)

struct TabView {
  const float2* coef;      // [sum_s nseg_s][TAB_NF][TAB_NC] coefficients (hi, lo), c_0 halved;
                           //   functions S, h, tau, dS/dtheta, dh/dtheta
  const int64_t* seg0;     // [S] first segment of spectrum s
  const int32_t* nseg;     // [S] segments of spectrum s
  const double* lo;        // [S] table origin: the spectrum's lower bound
};

// Granules of a spectrum: the samples in runs of GRANULE, from its first sample k0; the
// runs of spectrum s start at granule_base(k0, s) (no two spectra overlap: a spectrum has
// at most one run more than its samples fill).
constexpr int GRANULE = 32;
__host__ __device__ constexpr int64_t granule_base(int64_t k0, int64_t s) { return k0 / GRANULE + s; }
__host__ __device__ constexpr int64_t granule_count(int64_t n_samples, int64_t S) { return n_samples / GRANULE + S; }

struct EvalArgs {
  const Unit* units;
  int32_t n_units;
  const double* theta;     // [Q][nmax] log10 tau
  // Samples for the column sums, float-float {high, high, low, low} of one quantity per
  // plane: kq0 (omega 2^-30)^2, kq1 eps', kq2 omega eps''. Every part is stored twice so
  // that a 16-byte load gives both operands of the packed FP32 instructions.
  const float4* kq0;       // [sum K]
  const float4* kq1;       // [sum K]
  const float4* kq2;       // [sum K]
  // Per granule of a spectrum: {smallest (omega 2^-30)^2, largest eps', largest omega eps'',
  // largest (omega 2^-30)^2}; the second and third are infinite unless every eps' and
  // omega eps'' of the granule is finite and >= 0.
  const float4* kg;
  const double* omega;     // [sum K] FP64 inputs
  const double* eps_re;
  const double* eps_im;
  const double* h0;        // [S] sum_k eps'_k
  const double* bb;        // [S] b^T b = sum_k eps'_k^2 + eps''_k^2
  const uint8_t* active;   // [Q] optional candidate mask (nullptr: all)
  int32_t* n_failed;       // [S] optional: +1 per evaluated candidate whose damped matrix is not
                           //   positive definite (its cost is +inf)
  int32_t fuse_solve;      // column-sum pass: solve each unit's candidates (a warp each) as its sums are done
  int32_t sums_f64;        // column-sum pass: write tau and the sums in FP64 (the tables' node pass)
  int32_t ks;              // lanes per candidate in the pass kernels (power of two <= 32)
  double lam;
  double* out_cost;        // PH_SOLVE / PH_SOLVEG and fuse_solve outputs: cost [Q], weights [Q][nmax+1] or
  double* out_weights;     //   nullptr, gradient [Q][nmax] (PH_SOLVEG)
  double* out_grad;
  Scratch sc;
  TabView tab;             // DEBYE_PREC_MIXED_TABLE: the spectra's column-sum tables
  int* status;             // device status word
};

// ------------------------------------------------------------------ status word
__device__ __forceinline__ void set_status(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// Record the outcome of candidate q's factorisation (spectrum s).
__device__ __forceinline__ void record_fail(const EvalArgs& a, int q, int s, bool ok) {
  a.sc.fail[q] = ok ? 0 : 1;
  if (!ok && a.n_failed) atomicAdd(&a.n_failed[s], 1);
}

// ------------------------------------------------------------------ float-float helpers
// Error-free transformations (Dekker 1971; Knuth TAOCP vol. 2, 4.2.2). The
// __f*_rn intrinsics keep the compiler from contracting the rounded operations
// into FMAs, which would break the error terms.
__device__ __forceinline__ float rcp_approx(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}

// s + e == a + b exactly (Knuth TwoSum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// ------------------------------------------------------------------ packed FP32
// The column-sum pass runs its float-float steps on one pole (V = float) or on two poles
// at once (V = float2, the packed instructions of sm_100 and later: two IEEE operations,
// rounded as the scalar ones, for one issue slot; measured rate: half the issues of the
// scalar form at the same FP32 throughput). The v_* operations below are the same for both.
__device__ __forceinline__ float v_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float v_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float v_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float v_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float v_neg(float a) { return -a; }
__device__ __forceinline__ float v_rcp(float a) { return rcp_approx(a); }
__device__ __forceinline__ float2 v_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 v_sub(float2 a, float2 b) { return __fadd2_rn(a, v_neg(b)); }
__device__ __forceinline__ float2 v_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 v_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 v_rcp(float2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }
template <class V> __device__ __forceinline__ V v_all(float a);
template <> __device__ __forceinline__ float v_all<float>(float a) { return a; }
template <> __device__ __forceinline__ float2 v_all<float2>(float a) { return make_float2(a, a); }
// one of a sample's duplicated parts
__device__ __forceinline__ void v_part(float2 dup, float& v) { v = dup.x; }
__device__ __forceinline__ void v_part(float2 dup, float2& v) { v = dup; }
// (max, min) of 1 and a >= 0
__device__ __forceinline__ void v_order1(float a, float& big, float& small) {
  big = fmaxf(1.f, a);
  small = fminf(1.f, a);
}
__device__ __forceinline__ void v_order1(float2 a, float2& big, float2& small) {
  v_order1(a.x, big.x, small.x);
  v_order1(a.y, big.y, small.y);
}
// s + e == a + b exactly: TwoSum, or with ORDERED (the caller knows |a| >= |b|) Dekker's
// Fast2Sum, whose 3 operations give the same error term.
template <bool ORDERED, class V>
__device__ __forceinline__ void v_two_sum(V a, V b, V& s, V& e) {
  s = v_add(a, b);
  const V bb = v_sub(s, a);
  if constexpr (ORDERED) e = v_sub(b, bb);
  else e = v_add(v_sub(a, v_sub(s, bb)), v_sub(b, bb));
}

// acc (hi, lo) += a * b, a and b float-float (one Dot2 step: TwoProduct by FMA, exact
// sum of the leading part, low-order terms gathered in lo).
template <bool ORDERED, class V>
__device__ __forceinline__ void v_add_prod(V& ah, V& al, V xh, V xl, V yh, V yl) {
  const V p = v_mul(xh, yh);
  V pe = v_fma(xh, yh, v_neg(p));
  pe = v_fma(xh, yl, v_fma(xl, yh, pe));
  V s, e;
  v_two_sum<ORDERED>(ah, p, s, e);
  ah = s;
  al = v_add(al, v_add(e, pe));
}

// Float-float product (ph, pl) = (ah, al) * (bh, bl) to about 2^-46 relative.
template <class V>
__device__ __forceinline__ void v_mul_ff(V ah, V al, V bh, V bl, V& ph, V& pl) {
  ph = v_mul(ah, bh);
  pl = v_fma(ah, bh, v_neg(ph));
  pl = v_fma(ah, bl, v_fma(al, bh, pl));
}

// acc (hi, lo) += x, 0 <= xh <= acc_hi, x float-float (Fast2Sum, exact).
template <class V>
__device__ __forceinline__ void v_add_pos(V& ah, V& al, V xh, V xl) {
  const V s = v_add(ah, xh);
  al = v_add(al, v_add(v_sub(xh, v_sub(s, ah)), xl));
  ah = s;
}

// Float-float value (hi + lo, |lo| <= ulp(hi)/2 after normalisation) for the
// per-candidate small-system algebra of the mixed path.
struct ff {
  float h, l;
};
// Conversions between FP64 and float-float without the FP64 pipe: on this GPU every FP64
// operation, conversions included, holds a sub-partition's FP64 pipe for 64 cycles per
// warp, so splitting a double the plain way (two conversions to FP32, one back, one
// subtraction) costs 260 cycles, as much as 13 float-float multiply-adds. The integer forms
// below take about 15 instructions and give the same bits; values outside the stated
// exponent ranges (zeros, subnormal and huge values, infinities, NaN) take the plain way.
//
// (h, l): h the FP32 nearest v, l the FP32 nearest v - h.
__device__ __forceinline__ ff ff_of(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t e = (hi >> 20) & 0x7ffu;
  ff r;
  if (e - (1023u - 70u) <= 180u) {   // 2^-70 <= |v| < 2^111: every part is a normal FP32 value
    const uint32_t sign = hi & 0x80000000u;
    // round the 52-bit fraction to 23 bits, ties to even (the carry may reach the exponent)
    const uint64_t rb = (((uint64_t)hi << 32) | lo) + (0x0fffffffu + ((lo >> 29) & 1u));
    const uint32_t rlo = (uint32_t)rb, rhi = (uint32_t)(rb >> 32);
    r.h = __uint_as_float((__funnelshift_r(rlo, rhi, 29) - (896u << 23)) | sign);   // rebiased exponent
    // the remainder in units of 2^(exponent - 52), below 2^28 in magnitude
    const int d = (int)(lo - (rlo & 0xe0000000u));
    const uint32_t unit = (((hi & 0x7ff00000u) << 3) - (948u << 23)) | sign;
    r.l = __fmul_rn(__int2float_rn(d), __uint_as_float(unit));
  } else {
    r.h = __double2float_rn(v);
    r.l = __double2float_rn(v - (double)r.h);
  }
  return r;
}
// Entry i of a float-float scratch array (Scratch::x and Scratch::G in mixed precision).
__device__ __forceinline__ ff load_ff(const double* p, int64_t i) {
  const float2 v = reinterpret_cast<const float2*>(p)[i];
  return ff{v.x, v.y};
}
__device__ __forceinline__ void store_ff(double* p, int64_t i, ff v) {
  reinterpret_cast<float2*>(p)[i] = make_float2(v.h, v.l);
}
// A non-negative integer up to 2^30.
__device__ __forceinline__ ff ff_of_int(int v) {
  const float h = __int2float_rn(v);
  return ff{h, __int2float_rn(v - (int)h)};
}
// The plain forms behind the integer ones are calls, so that they are branched around: as
// predicated instructions they would hold the FP64 pipe even when not taken.
static __device__ __noinline__ double dbl_of_plain(float a) { return (double)a; }
// The FP64 value of an FP32 one.
__device__ __forceinline__ double dbl_of(float a) {
  const uint32_t b = __float_as_uint(a), m = b & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)   // normal
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + (896u << 20))), (int)(b << 29));
  if (m == 0) return __hiloint2double((int)b, 0);
  return dbl_of_plain(a);
}
// ff_of((double)a.h + (double)a.l) of a normalised a: the low part rounded to the last bit
// of the sum's FP64 value, by adding and removing a power of two whose last bit that is.
__device__ __forceinline__ ff ff_round53(ff a) {
  const uint32_t hb = __float_as_uint(a.h), lb = __float_as_uint(a.l);
  uint32_t e = hb & 0x7f800000u;
  if (e - (60u << 23) < (190u << 23)) {   // 2^-67 <= |h| < 2^123
    if ((hb & 0x007fffffu) == 0 && (int)(hb ^ lb) < 0 && a.l != 0.f) e -= 1u << 23;   // the sum lies below a power of two
    const float c = __uint_as_float((e - (29u << 23)) | (lb & 0x80000000u));
    if (fabsf(a.l) < fabsf(c)) a.l = __fsub_rn(__fadd_rn(a.l, c), c);
    return a;
  }
  const double v = (double)a.h + (double)a.l;
  a.h = __double2float_rn(v);
  a.l = __double2float_rn(v - (double)a.h);
  return a;
}
__device__ __forceinline__ double ff_dbl(ff a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ ff ff_sum(ff a, ff b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  e = __fadd_rn(e, __fadd_rn(a.l, b.l));
  const float h = __fadd_rn(s, e);
  return ff{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ ff ff_neg(ff a) { return ff{-a.h, -a.l}; }
__device__ __forceinline__ ff ff_prod(ff a, ff b) {
  float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e));
  const float h = __fadd_rn(p, e);
  return ff{h, __fsub_rn(e, __fsub_rn(h, p))};
}
// a / b: quotient q1 = a_h / b_h corrected by the float-float remainder a - q1 b.
// Both quotients multiply by the approximate reciprocal of b_h (rcp.approx, about
// 1 ulp): the float-float remainder carries q1's error, so a / b keeps ~2^-43.
__device__ __forceinline__ ff ff_quot(ff a, ff b) {
  const float rb = rcp_approx(b.h);
  const float q1 = __fmul_rn(a.h, rb);
  const ff r = ff_sum(a, ff_neg(ff_prod(ff{q1, 0.f}, b)));
  const float q2 = __fmul_rn(r.h, rb);
  const float h = __fadd_rn(q1, q2);
  return ff{h, __fsub_rn(q2, __fsub_rn(h, q1))};
}

// 1 / d in FP64 for d >= 1 (the Debye basis's denominator): one Newton-Raphson step in
// FP64 (two FMAs; Markstein, IBM J. Res. Dev. 34, 1990) from a float-float reciprocal good
// to 2^-44, which the FP32 and integer pipes form and assemble into a double. The step
// leaves 2^-88 before its rounding, so the result is the correctly rounded quotient unless
// that lies within 2^-88 of a tie (one operand in 2^35). The division operator costs 5 times
// 64 cycles of the FP64 pipe per warp, this 2 times. Arguments of 2^70 and more, infinite
// or NaN, and those within 2^-20 below a power of two (whose reciprocals 1 + j 2^-53 + j^2
// 2^-106 lie beside ties) or with the sum below in another binade take the operator.
__device__ __forceinline__ double rcp_ge1(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d);
  if (hi - 0x3ff00000u < (70u << 20) && (hi & 0xfffffu) != 0xfffffu) {
    const ff f = ff_of(d);
    const float r0 = rcp_approx(f.h);
    float e = __fmaf_rn(-f.h, r0, 1.0f);
    e = __fmaf_rn(-f.l, r0, e);
    const uint32_t rb = __float_as_uint(r0);
    // r0 e in units of r0's last FP64 bit, below 2^31 in magnitude (rcp.approx: 1 ulp)
    int m = __float2int_rn(__fmul_rn(__fmul_rn(r0, e), __uint_as_float((306u - (rb >> 23)) << 23)));
    const bool pow2 = (rb & 0x007fffffu) == 0 && m < 0;   // the sum lies below a power of two: half units
    if (pow2) m <<= 1;
    const long long b0 = (long long)(((uint64_t)((rb >> 3) + (896u << 20)) << 32) | (rb << 29));
    const long long b = b0 + m;
    if (pow2 || (b ^ b0) >> 52 == 0) {
      const double y = __longlong_as_double(b);
      return __fma_rn(y, __fma_rn(-d, y, 1.0), y);
    }
  }
  return 1.0 / d;
}

// ------------------------------------------------------------------ SplitMix64
// Steele, Lea and Flood, "Fast splittable pseudorandom number generators",
// OOPSLA 2014: the SplitMix64 output function used as a key mixer.
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Key prefix over (seed, tag, spectrum, generation).
__host__ __device__ __forceinline__ uint64_t rng_prefix(uint64_t seed, uint64_t tag, uint64_t s,
                                                        uint64_t g) {
  uint64_t h = splitmix64(seed);
  h = splitmix64(h ^ tag);
  h = splitmix64(h ^ s);
  return splitmix64(h ^ g);
}

// Full 64-bit key for (prefix, particle, dim).
__host__ __device__ __forceinline__ uint64_t rng_key(uint64_t prefix, uint64_t p, uint64_t d) {
  return splitmix64(splitmix64(prefix ^ p) ^ d);
}

// Uniform double in [0, 1) for (prefix, particle, dim): the key's upper 53 bits.
__host__ __device__ __forceinline__ double rng_uniform(uint64_t prefix, uint64_t p, uint64_t d) {
  return (double)(rng_key(prefix, p, d) >> 11) * (1.0 / 9007199254740992.0);
}

// Integer in [0, m), m < 2^32: multiply-shift of the key's upper 32 bits (Lemire 2019,
// without rejection).
__host__ __device__ __forceinline__ uint32_t rng_below(uint64_t key, uint32_t m) {
  return (uint32_t)(((key >> 32) * (uint64_t)m) >> 32);
}

constexpr uint64_t TAG_INIT_POS = 1, TAG_INIT_VEL = 2, TAG_R1 = 3, TAG_R2 = 4;
// differential evolution: donor indices, forced coordinate, crossover, bound re-draw, F
constexpr uint64_t TAG_DE_IDX = 5, TAG_DE_J = 6, TAG_DE_CR = 7, TAG_DE_BOUND = 8, TAG_DE_F = 9;
// dual annealing: uniforms of the visiting deviates, acceptance draws
constexpr uint64_t TAG_DA_VISIT = 10, TAG_DA_ACCEPT = 11;

}  // namespace debyefit
