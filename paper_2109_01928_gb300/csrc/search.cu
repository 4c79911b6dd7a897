// Search kernels of libdebyefit: particle swarm and differential evolution
// (Sec. III-B), top-k selection, projected L-BFGS polish, final re-solve and
// result assembly.
//
// Swarm update order matches the reference arithmetic exactly: explicit
// __d*_rn operations (no FMA contraction) so that positions are bit-identical
// to an FP64 implementation evaluating
//   v = (omega v + (phi_p r1) (p - x)) + (phi_g r2) (g - x),  x = clip(x + v, lo, hi).
#include <climits>
#include <cmath>

#include "dmath.cuh"
#include "launch.h"
#include "search.h"

namespace debyefit {

// Spectrum field of the generator's key: the caller's index map, else the batch index.
__device__ __forceinline__ uint64_t key_id(const SwarmArgs& a, int64_t s) {
  return a.rng_id ? (uint64_t)a.rng_id[s] : (uint64_t)s;
}

__global__ void k_pso_init(SwarmArgs a) {
  const int64_t Q = (int64_t)a.S * a.P;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < Q;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = q / a.P, p = q % a.P;
    const int N = a.n_poles[s];
    const double lo = a.lo[s], hi = a.hi[s], span = __dsub_rn(hi, lo);
    const uint64_t pp = rng_prefix(a.seed, TAG_INIT_POS, key_id(a, s), 0);
    const uint64_t pv = rng_prefix(a.seed, TAG_INIT_VEL, key_id(a, s), 0);
    for (int d = 0; d < a.nmax; ++d) {
      double x = 0.0, v = 0.0;
      if (d < N) {
        x = __dadd_rn(lo, __dmul_rn(span, rng_uniform(pp, p, d)));
        v = __dadd_rn(-span, __dmul_rn(__dmul_rn(2.0, span), rng_uniform(pv, p, d)));
      }
      a.x[q * a.nmax + d] = x;
      a.v[q * a.nmax + d] = v;
    }
  }
}

// A draw's 53-bit integer u (the uniform is u 2^-53) as a double, built from its
// IEEE-754 fields with integer operations (exact for u < 2^53): on GB300 an FP64
// conversion costs as much as any other FP64 operation.
__device__ __forceinline__ double u53_double(uint64_t u) {
  if (u == 0) return 0.0;
  const int e = 63 - __clzll((long long)u);   // position of the top bit, 0..52
  const uint64_t mant = (u << (52 - e)) & 0x000FFFFFFFFFFFFFull;
  return __longlong_as_double((long long)(((uint64_t)(e + 1023) << 52) | mant));
}

// fmin(fmax(v, lo), hi) by integer comparisons (an FP64 one holds the FP64 pipe as long as
// an FP64 addition); with a NaN or infinite operand, the FP64 form.
__device__ __forceinline__ long long ordered_bits(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
// (calls, so that they are branched around: predicated, they would hold the pipe all the same)
static __device__ __noinline__ double clamp_plain(double v, double lo, double hi) { return fmin(fmax(v, lo), hi); }
static __device__ __noinline__ double mul_plain(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double clamp_to(double v, double lo, double hi) {
  if (!(finite_bits(v) && finite_bits(lo) && finite_bits(hi))) return clamp_plain(v, lo, hi);
  if (ordered_bits(v) < ordered_bits(lo)) v = lo;
  return ordered_bits(v) > ordered_bits(hi) ? hi : v;
}

// The swarm update's coefficients. phi r = phi (u 2^-53) = (phi 2^-53) u: the scaling by
// 2^-53 is exact, so both round the same exact product once and the update stays
// bit-identical to phi * r (for any |phi| >= 2^-969, where phi 2^-53 is still a normal
// number). A positive power of two (the defaults are 0.5) multiplies by adding to the
// exponent, off the FP64 pipe.
struct MoveCoef {
  double omega, cp, cg;
  int eo, ep, eg;   // exponents of omega, cp, cg if powers of two, else INT_MIN
  static __device__ __forceinline__ int pow2(double v) {
    const int hi = __double2hiint(v);
    return (hi & 0xfffff) == 0 && __double2loint(v) == 0 && hi > 0x00100000 && hi < 0x7fe00000 ? (hi >> 20) - 1023
                                                                                           : INT_MIN;
  }
  static __device__ __forceinline__ MoveCoef of(const SwarmArgs& a) {
    MoveCoef c;
    c.omega = a.omega;
    c.cp = __dmul_rn(a.phi_p, 0x1p-53);
    c.cg = __dmul_rn(a.phi_g, 0x1p-53);
    c.eo = pow2(c.omega);
    c.ep = pow2(c.cp);
    c.eg = pow2(c.cg);
    return c;
  }
  // c v, c = 2^e where e != INT_MIN: exact unless the product leaves the normal range
  static __device__ __forceinline__ double mul(double c, int e, double v) {
    const int hi = __double2hiint(v), ev = (hi >> 20) & 0x7ff;
    if (e != INT_MIN && ev != 0 && ev != 0x7ff && ev + e > 0 && ev + e < 0x7ff)
      return __hiloint2double(hi + (e << 20), __double2loint(v));
    return mul_plain(c, v);
  }
};

// One coordinate: new velocity (returned) and position of x.
__device__ __forceinline__ double move_one(const MoveCoef& c, uint64_t key1, uint64_t key2, double& x, double v,
                                           double pb, double gb, double lo, double hi) {
  const double u1 = u53_double(key1 >> 11), u2 = u53_double(key2 >> 11);
  const double t1 = MoveCoef::mul(c.omega, c.eo, v);
  const double t2 = __dmul_rn(MoveCoef::mul(c.cp, c.ep, u1), __dsub_rn(pb, x));
  const double t3 = __dmul_rn(MoveCoef::mul(c.cg, c.eg, u2), __dsub_rn(gb, x));
  const double vn = __dadd_rn(__dadd_rn(t1, t2), t3);
  x = clamp_to(__dadd_rn(x, vn), lo, hi);
  return vn;
}

// One thread per coordinate of a spectrum's swarm: rows are read and written contiguously
// (a thread per particle strode through its row, re-reading every sector up to 4 times),
// and the keys' prefixes, the same for a whole spectrum, are formed once per block. What is
// left is the FP64 pipe: 7 operations per coordinate (10 with coefficients that are no
// powers of two), 64 cycles per warp each. 1024 spectra x 256 particles, N 2-12: 83 -> 57
// us. It serves what pso_step_fused turns away.
constexpr int MOVE_BLOCK = 256;
__global__ void __launch_bounds__(MOVE_BLOCK) k_pso_move(SwarmArgs a, int chunks) {
  __shared__ uint64_t prefix[2];
  const int gen = *a.gen;
  const int rows = (a.P + chunks - 1) / chunks;   // particles of a block's turn
  const MoveCoef co = MoveCoef::of(a);
  for (int64_t w = blockIdx.x; w < a.S * chunks; w += gridDim.x) {
    const int64_t s = w / chunks;
    const int p0 = (int)(w % chunks) * rows, p1 = min(a.P, p0 + rows);
    if (threadIdx.x < 2)
      prefix[threadIdx.x] = rng_prefix(a.seed, threadIdx.x ? TAG_R2 : TAG_R1, key_id(a, s), (uint64_t)gen);
    __syncthreads();
    const int N = a.n_poles[s];
    const double lo = a.lo[s], hi = a.hi[s];
    const int64_t row0 = s * a.P;
    const double* best = a.pbx + (row0 + a.gbest[s]) * a.nmax;
    for (int e = p0 * N + (int)threadIdx.x; e < p1 * N; e += MOVE_BLOCK) {
      const int p = e / N, d = e - p * N;
      const int64_t at = (row0 + p) * a.nmax + d;
      double x = a.x[at];
      a.v[at] = move_one(co, rng_key(prefix[0], p, d), rng_key(prefix[1], p, d), x, a.v[at], a.pbx[at], best[d], lo, hi);
      a.x[at] = x;
    }
    __syncthreads();   // the prefixes are read before the next turn's are written
  }
}

// Differential evolution (Storn and Price): one trial vector per population member.
// The population lives in pbx/pbc (k_pso_best's strictly-lower replacement is
// the evolution's selection), the trials are written to x for evaluation.
//   donors: slot j draws r below P-1-j and takes the r-th free index (ascending),
//           free = not the target and not an earlier slot;
//   mutant: rand/1  x_r0 + F (x_r1 - x_r2)   best/1  x_best + F (x_r0 - x_r1),
//           F = f_lo + (f_hi - f_lo) u once per generation;
//   a mutant coordinate outside [lo, hi] is re-drawn uniformly in the box;
//   binomial crossover: coordinate d from the mutant if u_d < CR or d = j_rand.
// Explicit __d*_rn operations keep the trials bit-identical to an FP64
// implementation evaluating the same expressions.
__global__ void k_de_trial(SwarmArgs a) {
  const int64_t Q = (int64_t)a.S * a.P;
  const int gen = *a.gen;
  const int k = a.de_strategy == DEBYE_DE_RAND1 ? 3 : 2;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < Q;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = q / a.P;
    const int p = (int)(q % a.P);
    const int N = a.n_poles[s];
    const double lo = a.lo[s], hi = a.hi[s], span = __dsub_rn(hi, lo);
    const uint64_t pidx = rng_prefix(a.seed, TAG_DE_IDX, key_id(a, s), (uint64_t)gen);
    const uint64_t pj = rng_prefix(a.seed, TAG_DE_J, key_id(a, s), (uint64_t)gen);
    const uint64_t pcr = rng_prefix(a.seed, TAG_DE_CR, key_id(a, s), (uint64_t)gen);
    const uint64_t pb = rng_prefix(a.seed, TAG_DE_BOUND, key_id(a, s), (uint64_t)gen);
    const double uf = rng_uniform(rng_prefix(a.seed, TAG_DE_F, key_id(a, s), (uint64_t)gen), 0, 0);
    const double F = __dadd_rn(a.de_f_lo, __dmul_rn(__dsub_rn(a.de_f_hi, a.de_f_lo), uf));
    int taken[4];  // sorted ascending
    int r[3] = {0, 0, 0};
    taken[0] = p;
    int nt = 1;
    for (int j = 0; j < k; ++j) {
      int v = (int)rng_below(rng_key(pidx, (uint64_t)p, (uint64_t)j), (uint32_t)(a.P - 1 - j));
      for (int t = 0; t < nt; ++t) v += (v >= taken[t]) ? 1 : 0;
      r[j] = v;
      int t = nt++;
      while (t > 0 && taken[t - 1] > v) {
        taken[t] = taken[t - 1];
        --t;
      }
      taken[t] = v;
    }
    const int64_t base = s * a.P + (k == 3 ? r[0] : a.gbest[s]);
    const int64_t d1 = s * a.P + (k == 3 ? r[1] : r[0]);
    const int64_t d2 = s * a.P + (k == 3 ? r[2] : r[1]);
    const int jr = (int)rng_below(rng_key(pj, (uint64_t)p, 0), (uint32_t)N);
    for (int d = 0; d < N; ++d) {
      double v = __dadd_rn(a.pbx[base * a.nmax + d],
                           __dmul_rn(F, __dsub_rn(a.pbx[d1 * a.nmax + d], a.pbx[d2 * a.nmax + d])));
      if (v < lo || v > hi) v = __dadd_rn(lo, __dmul_rn(span, rng_uniform(pb, (uint64_t)p, (uint64_t)d)));
      const bool take = rng_uniform(pcr, (uint64_t)p, (uint64_t)d) < a.de_cr || d == jr;
      a.x[q * a.nmax + d] = take ? v : a.pbx[q * a.nmax + d];
    }
  }
}

// ------------------------------------------------------------------ dual annealing
// Generalized simulated annealing chains (Tsallis and Stariolo), one per member:
// current state in cx/ce, best state in pbx/pbc, trial states written to x for
// evaluation. Outer iteration t (the device generation counter) has visiting
// temperature T(t) = T0 (2^(qv-1) - 1) / ((1+t)^(qv-1) - 1) and acceptance
// temperature T(t)/t; its Markov chain has 2N moves, move j < N displacing every
// coordinate and move j >= N coordinate j - N, by dx = sigma(T) z1 / |z2|^a with
// a = (qv-1)/(3-qv), sigma(T) = exp((log T - C_QV) / (3-qv)) and (z1, z2) a
// polar-method normal pair (capped at |dx| <= 1e8), wrapped periodically into
// [lo, hi]. A lower energy is accepted; a higher one with probability
// [1 - (1-qa) dE / T_acc]^(1/(1-qa)) against a uniform draw. All arithmetic is
// explicit __d*_rn and the fixed-operation log/exp, so the chains are
// bit-identical to an FP64 implementation of the same sequence.
constexpr double DA_QV = 2.62;
constexpr double DA_C_QV = -0.6233798028078907;  // (qv-1) log(A/B) at qv = 2.62 (40-digit evaluation)
constexpr double DA_TAIL = 1.0e8;
constexpr int DA_NMAX_SLOTS = 20;                // slot stride per move (pole capacity)

__device__ __forceinline__ double da_temperature(double t0, int t) {
  const double num = __dsub_rn(dm_exp(__dmul_rn(__dsub_rn(DA_QV, 1.0), dm_log(2.0))), 1.0);
  const double den = __dsub_rn(dm_exp(__dmul_rn(__dsub_rn(DA_QV, 1.0), dm_log(__dadd_rn((double)t, 1.0)))), 1.0);
  return __ddiv_rn(__dmul_rn(t0, num), den);
}

// Copy the evaluated initial members into the chains' current states.
__global__ void k_da_start(SwarmArgs a) {
  const int64_t Q = (int64_t)a.S * a.P;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < Q;
       q += (int64_t)gridDim.x * blockDim.x) {
    for (int d = 0; d < a.nmax; ++d) a.cx[q * a.nmax + d] = a.pbx[q * a.nmax + d];
    a.ce[q] = a.pbc[q];
  }
}

__global__ void k_da_visit(SwarmArgs a, int j) {
  const int64_t Q = (int64_t)a.S * a.P;
  const int t = *a.gen;
  const double T = da_temperature(a.da_t0, t);
  const double sig = dm_exp(__ddiv_rn(__dsub_rn(dm_log(T), DA_C_QV), __dsub_rn(3.0, DA_QV)));
  const double pw = __ddiv_rn(__dsub_rn(DA_QV, 1.0), __dsub_rn(3.0, DA_QV));
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < Q;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = q / a.P;
    const int p = (int)(q % a.P);
    const int N = a.n_poles[s];
    if (j >= 2 * N) {
      a.active[q] = 0;
      continue;
    }
    a.active[q] = 1;
    const double lo = a.lo[s], hi = a.hi[s], span = __dsub_rn(hi, lo);
    const uint64_t pv = rng_prefix(a.seed, TAG_DA_VISIT, key_id(a, s), (uint64_t)t);
    const int d0 = j < N ? 0 : j - N, d1 = j < N ? N : j - N + 1;
    for (int d = 0; d < a.nmax; ++d) {
      double xv = a.cx[q * a.nmax + d];
      if (d >= d0 && d < d1) {
        double z1 = 0.0, z2 = 0.0;
        for (int k = 0; k < DM_POLAR_TRIES; ++k) {
          const uint64_t slot = ((uint64_t)(j * DA_NMAX_SLOTS + d) * DM_POLAR_TRIES + k) * 2;
          const double u = __dsub_rn(__dmul_rn(2.0, rng_uniform(pv, (uint64_t)p, slot)), 1.0);
          const double v = __dsub_rn(__dmul_rn(2.0, rng_uniform(pv, (uint64_t)p, slot + 1)), 1.0);
          const double ss = __dadd_rn(__dmul_rn(u, u), __dmul_rn(v, v));
          if (ss > 0.0 && ss < 1.0) {
            const double f = __dsqrt_rn(__ddiv_rn(__dmul_rn(-2.0, dm_log(ss)), ss));
            z1 = __dmul_rn(u, f);
            z2 = __dmul_rn(v, f);
            break;
          }
        }
        const double az = fabs(z2);
        double dx;
        if (az > 0.0) dx = __ddiv_rn(__dmul_rn(sig, z1), dm_exp(__dmul_rn(pw, dm_log(az))));
        else dx = copysign(DA_TAIL, z1);
        dx = fmin(fmax(dx, -DA_TAIL), DA_TAIL);
        xv = __dadd_rn(xv, dx);
        if (xv < lo || xv > hi) {
          double r = fmod(__dsub_rn(xv, lo), span);
          if (r < 0.0) r = __dadd_rn(r, span);
          xv = __dadd_rn(lo, r);
        }
      }
      a.x[q * a.nmax + d] = xv;
    }
  }
}

__global__ void k_da_accept(SwarmArgs a, const double* __restrict__ cost, int j) {
  const int64_t Q = (int64_t)a.S * a.P;
  const int t = *a.gen;
  const double T = da_temperature(a.da_t0, t);
  const double t_acc = __ddiv_rn(T, (double)t);
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < Q;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = q / a.P;
    const int p = (int)(q % a.P);
    const int N = a.n_poles[s];
    if (j >= 2 * N) continue;
    double et = cost[q];
    if (!isfinite(et)) et = INFINITY;
    const double e = a.ce[q];
    bool acc = et < e;
    if (!acc && isfinite(et)) {
      const double tmp = __dsub_rn(1.0, __ddiv_rn(__dmul_rn(__dsub_rn(1.0, a.da_qa), __dsub_rn(et, e)), t_acc));
      const double pr = tmp > 0.0 ? dm_exp(__ddiv_rn(dm_log(tmp), __dsub_rn(1.0, a.da_qa))) : 0.0;
      const double u = rng_uniform(rng_prefix(a.seed, TAG_DA_ACCEPT, key_id(a, s), (uint64_t)t), (uint64_t)p,
                                   (uint64_t)j);
      acc = u <= pr;
    }
    if (!acc) continue;
    for (int d = 0; d < N; ++d) a.cx[q * a.nmax + d] = a.x[q * a.nmax + d];
    a.ce[q] = et;
    if (et < a.pbc[q]) {
      for (int d = 0; d < N; ++d) a.pbx[q * a.nmax + d] = a.x[q * a.nmax + d];
      a.pbc[q] = et;
    }
  }
}

// Lexicographic (cost, index) minimum: lowest cost, lowest index on ties.
__device__ __forceinline__ void argmin_merge(double& c, int& i, double c2, int i2) {
  if (c2 < c || (c2 == c && i2 < i)) {
    c = c2;
    i = i2;
  }
}
// The same on a cost's ordered bits (no NaN; a negative zero as a positive one).
__device__ __forceinline__ long long cost_key(double c) {
  const long long b = __double_as_longlong(c);
  return b == (long long)0x8000000000000000ull ? 0 : ordered_bits(c);
}
__device__ __forceinline__ void argmin_merge(long long& c, int& i, long long c2, int i2) {
  if (c2 < c || (c2 == c && i2 < i)) {
    c = c2;
    i = i2;
  }
}

__device__ __forceinline__ void block_argmin(double& c, int& i) {
  __shared__ double sc[32];
  __shared__ int si[32];
  for (int o = 16; o > 0; o >>= 1) {
    const double c2 = __shfl_down_sync(0xffffffffu, c, o);
    const int i2 = __shfl_down_sync(0xffffffffu, i, o);
    argmin_merge(c, i, c2, i2);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    sc[wid] = c;
    si[wid] = i;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    c = lane < nw ? sc[lane] : INFINITY;
    i = lane < nw ? si[lane] : 0x7fffffff;
    for (int o = 16; o > 0; o >>= 1) {
      const double c2 = __shfl_down_sync(0xffffffffu, c, o);
      const int i2 = __shfl_down_sync(0xffffffffu, i, o);
      argmin_merge(c, i, c2, i2);
    }
  }
  __syncthreads();
}

// Personal bests (strictly lower cost replaces; generation 0 initialises) and
// the global best per spectrum; one block per spectrum.
__global__ void k_pso_best(SwarmArgs a, const double* __restrict__ cost) {
  const int gen = *a.gen;
  for (int64_t s = blockIdx.x; s < a.S; s += gridDim.x) {
    const int N = a.n_poles[s];
    double bc = INFINITY;
    int bi = 0x7fffffff;
    for (int p = threadIdx.x; p < a.P; p += blockDim.x) {
      const int64_t q = s * a.P + p;
      double c = cost[q];
      if (!isfinite(c)) c = INFINITY;
      double pc = a.pbc[q];
      if (gen == 0 || c < pc) {
        pc = c;
        a.pbc[q] = c;
        for (int d = 0; d < N; ++d) a.pbx[q * a.nmax + d] = a.x[q * a.nmax + d];
      }
      argmin_merge(bc, bi, pc, p);
    }
    block_argmin(bc, bi);
    if (threadIdx.x == 0) {
      a.gbest[s] = bi < a.P ? bi : 0;
      if (a.trace) a.trace[s * (int64_t)(a.iters + 1) + gen] = bc;
      if (a.evals) atomicAdd(a.evals, (double)a.P * (double)(a.offsets[s + 1] - a.offsets[s]));
    }
  }
}

// k_pso_best and the move of the next generation in one kernel, one block per spectrum: the
// bests and the move read the same rows, and a generation of a small batch is bound by the
// launches' latencies (one spectrum of 64 particles: 13.4 us for the two, with the counter's
// kernel, against 6.8; 1024 spectra x 256: 73 against 50); where a spectrum has more work
// than that, pso_step_fused. The generation just evaluated is gens[s], advanced by the
// spectrum's own block. Improved rows are copied to the personal bests as the move passes
// over them; the global best's row is taken to shared memory first, since its particle
// moves too.
constexpr int STEP_BLOCK = 256;
template <bool MOVE>
__global__ void __launch_bounds__(STEP_BLOCK) k_pso_step(SwarmArgs a, const double* __restrict__ cost) {
  __shared__ uint64_t prefix[2];
  __shared__ double best[NMAX];
  __shared__ unsigned char improved[PSO_STEP_MAX_P];
  __shared__ long long red_c[STEP_BLOCK / 32];
  __shared__ int red_i[STEP_BLOCK / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const MoveCoef co = MoveCoef::of(a);
  for (int64_t s = blockIdx.x; s < a.S; s += gridDim.x) {
    const int gen = a.gens[s], N = a.n_poles[s];
    const int64_t row0 = s * a.P;
    if (MOVE && threadIdx.x >= STEP_BLOCK - 2) {   // the last warp's lanes: the others reduce meanwhile
      const int k = threadIdx.x & 1;
      prefix[k] = rng_prefix(a.seed, k ? TAG_R2 : TAG_R1, key_id(a, s), (uint64_t)(gen + 1));
    }
    // personal bests (strictly lower cost replaces; generation 0 initialises) and the best particle
    long long bc = 0x7ff0000000000000ll;   // +infinity
    int bi = 0x7fffffff;
    for (int p = threadIdx.x; p < a.P; p += STEP_BLOCK) {
      double c = cost[row0 + p];
      if (!finite_bits(c)) c = INFINITY;
      long long kc = cost_key(c);
      const long long kp = gen == 0 ? 0 : cost_key(a.pbc[row0 + p]);
      const bool better = gen == 0 || kc < kp;
      if (better) a.pbc[row0 + p] = c;
      else kc = kp;
      improved[p] = better;
      argmin_merge(bc, bi, kc, p);
    }
    for (int o = 16; o > 0; o >>= 1) {
      const long long c2 = __shfl_xor_sync(0xffffffffu, bc, o);
      const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
      argmin_merge(bc, bi, c2, i2);
    }
    if (lane == 0) {
      red_c[wid] = bc;
      red_i[wid] = bi;
    }
    __syncthreads();
    bc = red_c[0];
    bi = red_i[0];
#pragma unroll
    for (int w = 1; w < STEP_BLOCK / 32; ++w) argmin_merge(bc, bi, red_c[w], red_i[w]);
    const int gi = bi < a.P ? bi : 0;
    if (threadIdx.x < N) {
      const int64_t at = (row0 + gi) * a.nmax + threadIdx.x;
      best[threadIdx.x] = improved[gi] ? a.x[at] : a.pbx[at];
    }
    if (threadIdx.x == 0) {
      a.gbest[s] = gi;
      a.gens[s] = gen + 1;
      // the best cost itself: +infinity if there is none
      if (a.trace) a.trace[s * (int64_t)(a.iters + 1) + gen] = bi < a.P ? a.pbc[row0 + gi] : INFINITY;
      if (a.evals && s == 0) atomicAdd(a.evals, (double)a.P * (double)(a.offsets[a.S] - a.offsets[0]));
    }
    __syncthreads();
    const double lo = a.lo[s], hi = a.hi[s];
    for (int e = threadIdx.x; e < a.P * N; e += STEP_BLOCK) {
      const int p = e / N, d = e - p * N;
      const int64_t at = (row0 + p) * a.nmax + d;
      const bool imp = improved[p];
      if (!MOVE && !imp) continue;
      double x = a.x[at];
      double pb = x;
      if (imp) a.pbx[at] = x;
      else pb = a.pbx[at];
      if (MOVE) {
        a.v[at] = move_one(co, rng_key(prefix[0], p, d), rng_key(prefix[1], p, d), x, a.v[at], pb, best[d], lo, hi);
        a.x[at] = x;
      }
    }
    __syncthreads();   // shared state is free for the next spectrum
  }
}

// After an outer iteration of dual annealing: best chain per spectrum (lowest
// best cost, lowest index on ties), its cost in the trace, and the iteration's
// evaluations (P chains x 2N moves x K samples) in the counter.
__global__ void k_da_best(SwarmArgs a) {
  const int gen = *a.gen;
  for (int64_t s = blockIdx.x; s < a.S; s += gridDim.x) {
    double bc = INFINITY;
    int bi = 0x7fffffff;
    for (int p = threadIdx.x; p < a.P; p += blockDim.x) argmin_merge(bc, bi, a.pbc[s * a.P + p], p);
    block_argmin(bc, bi);
    if (threadIdx.x == 0) {
      a.gbest[s] = bi < a.P ? bi : 0;
      if (a.trace) a.trace[s * (int64_t)(a.iters + 1) + gen] = bc;
      if (a.evals)
        atomicAdd(a.evals, (double)a.P * 2.0 * (double)a.n_poles[s] * (double)(a.offsets[s + 1] - a.offsets[s]));
    }
  }
}

__global__ void k_gen_advance(int* gen) { *gen += 1; }

__global__ void k_add_scalar(double* dst, double v) { *dst += v; }

// ------------------------------------------------------------------ top-k and polish
// Lines l = s * T + j start from the j-th best personal best of spectrum s.
__global__ void k_topk(SwarmArgs a, PolishArgs pa) {
  extern __shared__ unsigned char taken_raw[];
  unsigned char* taken = taken_raw;
  for (int64_t s = blockIdx.x; s < a.S; s += gridDim.x) {
    for (int p = threadIdx.x; p < a.P; p += blockDim.x) taken[p] = 0;
    __syncthreads();
    for (int j = 0; j < pa.T; ++j) {
      double bc = INFINITY;
      int bi = 0x7fffffff;
      for (int p = threadIdx.x; p < a.P; p += blockDim.x)
        if (!taken[p]) argmin_merge(bc, bi, a.pbc[s * a.P + p], p);
      block_argmin(bc, bi);
      if (threadIdx.x == 0) {
        const int p = bi < a.P ? bi : 0;
        taken[p] = 1;
        const int64_t l = s * pa.T + j;
        for (int d = 0; d < a.nmax; ++d) pa.th[l * a.nmax + d] = a.pbx[(s * a.P + p) * a.nmax + d];
        pa.f[l] = bc;
        pa.done[l] = 0;
        pa.hcount[l] = 0;
        pa.head[l] = 0;
        pa.acc[l] = 0;
      }
      __syncthreads();
    }
  }
}

// The start point of each line is evaluated, with its gradient, in the
// accepted-point slot (candidate l of the gradient evaluation).
__global__ void k_polish_start(PolishArgs pa) {
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < pa.L;
       l += (int64_t)gridDim.x * blockDim.x) {
    for (int d = 0; d < pa.nmax; ++d) pa.ath[l * pa.nmax + d] = pa.th[l * pa.nmax + d];
    pa.aactive[l] = 1;
    for (int t = 0; t < pa.R; ++t) pa.active[l * pa.R + t] = 0;
  }
}

// After the start evaluation: f, g of each line.
__global__ void k_polish_take0(PolishArgs pa) {
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < pa.L;
       l += (int64_t)gridDim.x * blockDim.x) {
    pa.f[l] = pa.acost[l];
    for (int d = 0; d < pa.nmax; ++d) pa.g[l * pa.nmax + d] = pa.agrad[l * pa.nmax + d];
    pa.aactive[l] = 0;
    if (!isfinite(pa.f[l])) pa.done[l] = 1;
  }
}

__device__ __forceinline__ double dotn(const double* a, const double* b, int n) {
  double s = 0.0;
  for (int i = 0; i < n; ++i) s = fma(a[i], b[i], s);
  return s;
}

// The line's next round of trials, t0 .. t0 + R - 1, by the lanes of its group.
__device__ void write_trials(const PolishArgs& pa, int64_t l, int N, double lo, double hi, int t0, int lane,
                             int group) {
  const int nmax = pa.nmax;
  for (int t = lane; t < pa.R; t += group) pa.active[l * pa.R + t] = t0 + t < pa.max_trials;
  const int live = min(pa.R, pa.max_trials - t0);
  for (int e = lane; e < live * nmax; e += group) {
    const int t = e / nmax, d = e - t * nmax;
    const double step = __hiloint2double((1023 - (t0 + t)) << 20, 0);   // 2^-(t0 + t)
    double v = 0.0;
    if (d < N) v = clamp_to(pa.th[l * nmax + d] + step * pa.dir[l * nmax + d], lo, hi);
    pa.tth[(l * pa.R + t) * nmax + d] = v;
  }
}

// The polish's per-line kernels run one thread per line through a dependent FP64 chain
// (the L-BFGS two-loop recursion, the Armijo tests): single-warp blocks spread the lines
// over every SM.
constexpr int POLISH_BLOCK = 32;

// dst += the warp's sum of v: evaluation counts, whole numbers, so the order of the sum is
// free, and one addition per warp replaces one per line on the same address (1024 spectra x
// 8 lines: 41 -> 30 us for the full steps' Armijo test).
__device__ __forceinline__ void add_count(double* dst, int64_t v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(dst, (double)v);
}

// L-BFGS update with the accepted point's cost and gradient: history pair (s, y) kept
// only when s^T y > eps y^T y (the oldest pair's slot taken over when full). The pair's rho
// and gamma, the same dot products that the recursion needs, are kept with it.
__device__ void polish_take(const PolishArgs& pa, int64_t l, int N) {
  const int nmax = pa.nmax, m = pa.m;
  pa.aactive[l] = 0;
  double sv[NMAX], yv[NMAX];
  for (int d = 0; d < N; ++d) {
    sv[d] = pa.ath[l * nmax + d] - pa.th[l * nmax + d];
    yv[d] = pa.agrad[l * nmax + d] - pa.g[l * nmax + d];
  }
  const double sy = dotn(sv, yv, N), yy = dotn(yv, yv, N);
  if (sy > 2.220446049250313e-16 * yy) {
    int hc = pa.hcount[l], head = pa.head[l];
    int slot = head + hc;
    if (slot >= m) slot -= m;
    if (hc == m) {
      slot = head;
      pa.head[l] = head + 1 == m ? 0 : head + 1;
    } else {
      pa.hcount[l] = hc + 1;
    }
    for (int d = 0; d < N; ++d) {
      pa.hs[(slot * nmax + d) * pa.L + l] = sv[d];
      pa.hy[(slot * nmax + d) * pa.L + l] = yv[d];
    }
    pa.rho[slot * pa.L + l] = 1.0 / sy;
    pa.gamma[l] = sy / yy;
  }
  for (int d = 0; d < N; ++d) {
    pa.th[l * nmax + d] = pa.ath[l * nmax + d];
    pa.g[l * nmax + d] = pa.agrad[l * nmax + d];
  }
  pa.f[l] = pa.acost[l];
  if (!isfinite(pa.f[l])) pa.done[l] = 1;
}

// Two-loop recursion (Nocedal and Wright, Alg. 7.4) for the direction d = -H g;
// a non-descent direction is replaced by -g / max(1, |g|_inf) and the history cleared.
__device__ void polish_dir(const PolishArgs& pa, int64_t l, int N, double lo, double hi) {
  const int nmax = pa.nmax, m = pa.m;
  double q[NMAX], alpha[8];
  const double* g = pa.g + l * nmax;
  for (int d = 0; d < N; ++d) q[d] = g[d];
  const int hc = pa.hcount[l], head = pa.head[l];
  auto slot = [&](int k) { return head + k >= m ? head + k - m : head + k; };   // k-th oldest pair
  const int64_t L = pa.L;
  for (int k = hc - 1; k >= 0; --k) {
    const double* sk = pa.hs + slot(k) * nmax * L + l;
    const double* yk = pa.hy + slot(k) * nmax * L + l;
    double dot = 0.0;
#pragma unroll 4
    for (int d = 0; d < N; ++d) dot = fma(sk[d * L], q[d], dot);
    const double al = pa.rho[slot(k) * L + l] * dot;
#pragma unroll 4
    for (int d = 0; d < N; ++d) q[d] -= al * yk[d * L];
    alpha[k] = al;
  }
  double gamma;
  if (hc > 0) {
    gamma = pa.gamma[l];
  } else {
    double gi = 0.0;
    for (int d = 0; d < N; ++d) gi = fmax(gi, fabs(g[d]));
    gamma = 1.0 / fmax(1.0, gi);
  }
  for (int d = 0; d < N; ++d) q[d] *= gamma;
  for (int k = 0; k < hc; ++k) {
    const double* sk = pa.hs + slot(k) * nmax * L + l;
    const double* yk = pa.hy + slot(k) * nmax * L + l;
    double dot = 0.0;
#pragma unroll 4
    for (int d = 0; d < N; ++d) dot = fma(yk[d * L], q[d], dot);
    const double be = pa.rho[slot(k) * L + l] * dot;
#pragma unroll 4
    for (int d = 0; d < N; ++d) q[d] += sk[d * L] * (alpha[k] - be);
  }
  double gd = 0.0;
  for (int d = 0; d < N; ++d) gd = fma(g[d], -q[d], gd);
  double* dir = pa.dir + l * nmax;
  if (!(gd < 0.0)) {
    double gi = 0.0;
    for (int d = 0; d < N; ++d) gi = fmax(gi, fabs(g[d]));
    const double sc = 1.0 / fmax(1.0, gi);
    for (int d = 0; d < N; ++d) dir[d] = -g[d] * sc;
    pa.hcount[l] = 0;
    pa.head[l] = 0;
  } else {
    for (int d = 0; d < N; ++d) dir[d] = -q[d];
  }
  // the full step t = 0 is evaluated first, with its gradient, in the accepted-point slot;
  // the backtracking rounds start at t = 1 if it fails
  for (int d = 0; d < nmax; ++d) {
    double v = 0.0;
    if (d < N) v = clamp_to(pa.th[l * nmax + d] + dir[d], lo, hi);
    pa.ath[l * nmax + d] = v;
  }
  pa.aactive[l] = 1;
  pa.t0[l] = 1;
}

// Between two evaluations of a line's points: the update of the iteration that ends (take,
// for the lines that accepted a step) and the direction of the one that begins.
__global__ void __launch_bounds__(POLISH_BLOCK) k_polish_step(PolishArgs pa, const int32_t* n_poles,
                                                              const double* lo_, const double* hi_) {
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < pa.L;
       l += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = l / pa.T;
    const int N = n_poles[s];
    if (pa.acc[l]) polish_take(pa, l, N);
    pa.acc[l] = 0;
    if (!pa.done[l]) polish_dir(pa, l, N, lo_[s], hi_[s]);
  }
}

// The Armijo tests: a group of lanes per line, one lane per trial of a round (8, or a warp
// where a round takes every step length), so that a round's tests run side by side and its
// next trials are written by the whole group. With one thread per line the 8 x N trial
// coordinates of a rejecting line were one thread's serial FP64 work, and its whole warp's:
// 1024 spectra x 8 lines, 30 and 49 us for the two kernels, now 11 and 14.
__device__ __forceinline__ int polish_group(const PolishArgs& pa) { return pa.R <= 8 ? 8 : 32; }
__device__ __forceinline__ unsigned polish_group_mask(int group) {
  return group == 32 ? 0xffffffffu : 0xffu << (threadIdx.x & 24);
}
constexpr int ARMIJO_BLOCK = 128;

// The full step (evaluated with its gradient in the accepted-point slot): accepted, the
// line's cost and gradient are ready for the update; rejected, the backtracking trials t =
// 1 .. R of the first round are written.
__global__ void __launch_bounds__(ARMIJO_BLOCK) k_polish_first(PolishArgs pa, const int32_t* n_poles,
                                                               const double* lo_, const double* hi_,
                                                               const int64_t* offsets) {
  const int group = polish_group(pa), lane = (int)threadIdx.x & (group - 1);
  const unsigned gmask = polish_group_mask(group);
  const int64_t step = (int64_t)gridDim.x * blockDim.x / group;
  int64_t evaluated = 0;
  for (int64_t l = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / group; l < pa.L; l += step) {
    const bool eval = pa.aactive[l];
    __syncwarp(gmask);   // every lane of the group has read the flag
    if (!eval) continue;
    const int64_t s = l / pa.T;
    const int N = n_poles[s];
    const int nmax = pa.nmax;
    double gs = 0.0;
    for (int d = 0; d < N; ++d) gs = fma(pa.g[l * nmax + d], pa.ath[l * nmax + d] - pa.th[l * nmax + d], gs);
    const bool ok = pa.acost[l] <= pa.f[l] + pa.c1 * gs;
    const int t0 = pa.t0[l];
    if (lane == 0) {
      evaluated += offsets[s + 1] - offsets[s];
      pa.aactive[l] = 0;
      if (ok) pa.acc[l] = 1;
      else if (t0 >= pa.max_trials) pa.done[l] = 1;
    }
    if (!ok && t0 < pa.max_trials) write_trials(pa, l, N, lo_[s], hi_[s], t0, lane, group);
  }
  __syncwarp();
  if (pa.evals) add_count(pa.evals, evaluated);
}

// The evaluated trials of each line, in order of decreasing step.
__global__ void __launch_bounds__(ARMIJO_BLOCK) k_polish_accept(PolishArgs pa, const int32_t* n_poles,
                                                                const double* lo_, const double* hi_,
                                                                const int64_t* offsets) {
  const int group = polish_group(pa), lane = (int)threadIdx.x & (group - 1);
  const unsigned gmask = polish_group_mask(group);
  const int64_t step = (int64_t)gridDim.x * blockDim.x / group;
  int64_t evaluated = 0;
  for (int64_t l = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / group; l < pa.L; l += step) {
    const bool skip = pa.done[l] || pa.acc[l];
    const int t0 = pa.t0[l];
    __syncwarp(gmask);   // every lane of the group has read the flags
    if (skip) continue;
    const int64_t s = l / pa.T, q = l * pa.R + lane;
    const int N = n_poles[s];
    const int nmax = pa.nmax;
    const bool act = lane < pa.R && pa.active[q];
    bool ok = false;
    if (act) {
      double gs = 0.0;
      for (int d = 0; d < N; ++d) gs = fma(pa.g[l * nmax + d], pa.tth[q * nmax + d] - pa.th[l * nmax + d], gs);
      ok = pa.tcost[q] <= pa.f[l] + pa.c1 * gs;
    }
    const int shift = __ffs((int)gmask) - 1;
    const unsigned oks = __ballot_sync(gmask, ok) >> shift, acts = __ballot_sync(gmask, act) >> shift;
    if (!acts) continue;
    // the trials a sequential backtracking search evaluates: up to and including the first
    // acceptable one (the speculative trials after it are not counted)
    const int hit = __ffs((int)oks) - 1;
    const int counted = hit >= 0 ? __popc(acts & ((2u << hit) - 1)) : __popc(acts);
    const bool more = hit < 0 && t0 + pa.R < pa.max_trials;
    if (lane == 0) {
      evaluated += counted * (offsets[s + 1] - offsets[s]);
      if (hit >= 0) {
        pa.aactive[l] = 1;
        pa.acc[l] = 1;
      } else {
        pa.t0[l] = t0 + pa.R;
        if (!more) pa.done[l] = 1;
      }
    }
    if (hit >= 0)
      for (int d = lane; d < nmax; d += group) pa.ath[l * nmax + d] = pa.tth[(l * pa.R + hit) * nmax + d];
    if (more) write_trials(pa, l, N, lo_[s], hi_[s], t0 + pa.R, lane, group);
    else if (lane < pa.R) pa.active[q] = 0;
  }
  __syncwarp();
  if (pa.evals) add_count(pa.evals, evaluated);
}

// The update of the last iteration.
__global__ void __launch_bounds__(POLISH_BLOCK) k_polish_take(PolishArgs pa, const int32_t* n_poles) {
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < pa.L;
       l += (int64_t)gridDim.x * blockDim.x)
    if (pa.acc[l]) polish_take(pa, l, n_poles[l / pa.T]);
}

// Best line per spectrum (lowest cost, lowest rank on ties), or the swarm's
// global best when there is no polish; writes theta* of spectrum s to out[s].
__global__ void k_pick_best(SwarmArgs a, PolishArgs pa, double* out_theta) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < a.S;
       s += (int64_t)gridDim.x * blockDim.x) {
    const double* src;
    if (pa.T > 0) {
      double bc = INFINITY;
      int bj = 0x7fffffff;
      for (int j = 0; j < pa.T; ++j) argmin_merge(bc, bj, pa.f[s * pa.T + j], j);
      if (bj >= pa.T) bj = 0;
      src = pa.th + (s * pa.T + bj) * a.nmax;
    } else {
      src = a.pbx + (s * a.P + a.gbest[s]) * a.nmax;
    }
    for (int d = 0; d < a.nmax; ++d) out_theta[s * a.nmax + d] = src[d];
  }
}

// Poles sorted by ascending tau (stable), padded with zeros (Listing 2 layout).
__global__ void k_assemble(int64_t S, int nmax, const int32_t* n_poles, const double* theta,
                           const double* weights, const double* cost, double* eps_inf, double* d_eps,
                           double* tau, double* final_cost) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int N = n_poles[s];
    int idx[NMAX];
    for (int i = 0; i < N; ++i) idx[i] = i;
    for (int i = 1; i < N; ++i) {
      const int v = idx[i];
      int j = i - 1;
      while (j >= 0 && theta[s * nmax + idx[j]] > theta[s * nmax + v]) {
        idx[j + 1] = idx[j];
        --j;
      }
      idx[j + 1] = v;
    }
    eps_inf[s] = weights[s * (nmax + 1)];
    for (int i = 0; i < nmax; ++i) {
      if (i < N) {
        d_eps[s * nmax + i] = weights[s * (nmax + 1) + 1 + idx[i]];
        tau[s * nmax + i] = exp10(theta[s * nmax + idx[i]]);
      } else {
        d_eps[s * nmax + i] = 0.0;
        tau[s * nmax + i] = 0.0;
      }
    }
    final_cost[s] = cost[s];
  }
}

// ------------------------------------------------------------------ launchers
static int g1d(int64_t n, int sms) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sms * 8)); }
// Grid for one thread per item in blocks of `block` threads (at most 2048 resident per SM).
static int g1d_b(int64_t n, int block, int sms) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + block - 1) / block, (int64_t)sms * (2048 / block)));
}

void launch_pso_init(const SwarmArgs& a, int sms, cudaStream_t st) {
  k_pso_init<<<g1d((int64_t)a.S * a.P, sms), 256, 0, st>>>(a);
}
void launch_pso_move(const SwarmArgs& a, int sms, cudaStream_t st) {
  // enough turns to fill the GPU, each of at least 16 particles
  const int64_t want = (int64_t)sms * 8;
  const int chunks = (int)std::max<int64_t>(1, std::min<int64_t>((want + a.S - 1) / a.S, (a.P + 15) / 16));
  k_pso_move<<<(int)std::min<int64_t>(a.S * chunks, (int64_t)sms * 32), MOVE_BLOCK, 0, st>>>(a, chunks);
}
void launch_de_trial(const SwarmArgs& a, int sms, cudaStream_t st) {
  k_de_trial<<<g1d((int64_t)a.S * a.P, sms), 256, 0, st>>>(a);
}
void launch_da_start(const SwarmArgs& a, int sms, cudaStream_t st) {
  k_da_start<<<g1d((int64_t)a.S * a.P, sms), 256, 0, st>>>(a);
}
void launch_da_visit(const SwarmArgs& a, int j, int sms, cudaStream_t st) {
  k_da_visit<<<g1d_b((int64_t)a.S * a.P, 128, sms), 128, 0, st>>>(a, j);
}
void launch_da_accept(const SwarmArgs& a, const double* cost, int j, int sms, cudaStream_t st) {
  k_da_accept<<<g1d((int64_t)a.S * a.P, sms), 256, 0, st>>>(a, cost, j);
}
void launch_da_best(const SwarmArgs& a, int sms, cudaStream_t st) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(a.S, (int64_t)sms * 8));
  k_da_best<<<grid, 256, 0, st>>>(a);
}
void launch_pso_best(const SwarmArgs& a, const double* cost, int sms, cudaStream_t st) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(a.S, (int64_t)sms * 8));
  k_pso_best<<<grid, 256, 0, st>>>(a, cost);
}
void launch_pso_step(const SwarmArgs& a, const double* cost, bool move, int sms, cudaStream_t st) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(a.S, (int64_t)sms * 8));
  if (move) k_pso_step<true><<<grid, STEP_BLOCK, 0, st>>>(a, cost);
  else k_pso_step<false><<<grid, STEP_BLOCK, 0, st>>>(a, cost);
}
void launch_gen_advance(int* gen, cudaStream_t st) { k_gen_advance<<<1, 1, 0, st>>>(gen); }
void launch_add_scalar(double* dst, double v, cudaStream_t st) { k_add_scalar<<<1, 1, 0, st>>>(dst, v); }
void launch_topk(const SwarmArgs& a, const PolishArgs& pa, int sms, cudaStream_t st) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(a.S, (int64_t)sms * 8));
  k_topk<<<grid, 256, a.P, st>>>(a, pa);
}
void launch_polish_start(const PolishArgs& pa, int sms, cudaStream_t st) {
  k_polish_start<<<g1d(pa.L, sms), 256, 0, st>>>(pa);
}
void launch_polish_take0(const PolishArgs& pa, int sms, cudaStream_t st) {
  k_polish_take0<<<g1d(pa.L, sms), 256, 0, st>>>(pa);
}
void launch_polish_step(const PolishArgs& pa, const int32_t* n_poles, const double* lo, const double* hi,
                        int sms, cudaStream_t st) {
  k_polish_step<<<g1d_b(pa.L, POLISH_BLOCK, sms), POLISH_BLOCK, 0, st>>>(pa, n_poles, lo, hi);
}
void launch_polish_first(const PolishArgs& pa, const int32_t* n_poles, const double* lo, const double* hi,
                         const int64_t* offsets, int sms, cudaStream_t st) {
  const int64_t lanes = pa.L * (pa.R <= 8 ? 8 : 32);
  k_polish_first<<<g1d_b(lanes, ARMIJO_BLOCK, sms), ARMIJO_BLOCK, 0, st>>>(pa, n_poles, lo, hi, offsets);
}
void launch_polish_accept(const PolishArgs& pa, const int32_t* n_poles, const double* lo, const double* hi,
                          const int64_t* offsets, int sms, cudaStream_t st) {
  const int64_t lanes = pa.L * (pa.R <= 8 ? 8 : 32);
  k_polish_accept<<<g1d_b(lanes, ARMIJO_BLOCK, sms), ARMIJO_BLOCK, 0, st>>>(pa, n_poles, lo, hi, offsets);
}
void launch_polish_take(const PolishArgs& pa, const int32_t* n_poles, int sms, cudaStream_t st) {
  k_polish_take<<<g1d_b(pa.L, POLISH_BLOCK, sms), POLISH_BLOCK, 0, st>>>(pa, n_poles);
}
void launch_pick_best(const SwarmArgs& a, const PolishArgs& pa, double* out_theta, int sms, cudaStream_t st) {
  k_pick_best<<<g1d(a.S, sms), 256, 0, st>>>(a, pa, out_theta);
}
void launch_assemble(int64_t S, int nmax, const int32_t* n_poles, const double* theta, const double* weights,
                     const double* cost, double* eps_inf, double* d_eps, double* tau, double* final_cost,
                     int sms, cudaStream_t st) {
  k_assemble<<<g1d(S, sms), 256, 0, st>>>(S, nmax, n_poles, theta, weights, cost, eps_inf, d_eps, tau,
                                           final_cost);
}

}  // namespace debyefit
