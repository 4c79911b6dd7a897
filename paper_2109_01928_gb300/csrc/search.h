// Device-side state of the particle swarm and the L-BFGS polish.
#pragma once
#include "common.cuh"

namespace debyefit {

struct SwarmArgs {
  int64_t S;
  int32_t P, nmax, iters;
  uint64_t seed;
  double omega, phi_p, phi_g;
  double de_f_lo, de_f_hi, de_cr;  // differential evolution coefficients
  int32_t de_strategy;             // DEBYE_DE_RAND1 or DEBYE_DE_BEST1
  double da_t0, da_qa;             // dual annealing: initial temperature, acceptance parameter
  const int32_t* n_poles;
  const double* lo;
  const double* hi;
  const int64_t* offsets;
  const int64_t* rng_id;  // [S] spectrum index used in the generator's keys, or nullptr (= s)
  double* x;       // [S*P][nmax] positions (log10 tau); differential evolution: trial vectors
  double* v;       // [S*P][nmax] velocities (swarm only)
  double* pbx;     // [S*P][nmax] personal-best positions; differential evolution: the population
  double* pbc;     // [S*P]       personal-best costs; differential evolution: population costs
  int32_t* gbest;  // [S]         global-best particle
  double* cx;      // [S*P][nmax] dual annealing: current chain states
  double* ce;      // [S*P]       dual annealing: current energies
  uint8_t* active; // [S*P]       dual annealing: member moved in this step (evaluation mask)
  int* gen;        // generation counter (device)
  int* gens;       // [S] generation counters of k_pso_step
  double* trace;   // [S][iters+1] or nullptr
  double* evals;   // [1] or nullptr
};

struct PolishArgs {
  int64_t L;       // lines = S * T
  int32_t T;       // lines per spectrum
  int32_t R;       // trial step lengths per backtracking round (after the full step)
  int32_t nmax, m, max_trials;
  double c1;
  double* th;      // [L][nmax] current point
  double* f;       // [L]
  double* g;       // [L][nmax]
  double* dir;     // [L][nmax]
  double* hs;      // [m][nmax][L] history s, a ring of pairs from slot head
  double* hy;      // [m][nmax][L] history y
  double* rho;     // [m][L] 1 / y^T s of each pair
  double* gamma;   // [L] s^T y / y^T y of the newest pair
  int32_t* hcount; // [L]
  int32_t* head;   // [L] slot of the oldest pair
  int32_t* t0;     // [L] first trial index of the next backtracking round
  int32_t* done;   // [L] line finished (no acceptable step or non-finite)
  int32_t* acc;    // [L] step accepted in this iteration (acost, agrad at ath ready after the last evaluation)
  double* tth;     // [L*R][nmax] trial points
  double* tcost;   // [L*R]
  uint8_t* active; // [L*R] trial needs evaluation
  // the accepted point of each line, evaluated with its gradient
  double* ath;     // [L][nmax] accepted point
  double* acost;   // [L]
  double* agrad;   // [L][nmax]
  uint8_t* aactive;// [L] ath needs a cost + gradient evaluation (the full step, or a later accepted trial)
  double* evals;   // [1] or nullptr
};

void launch_pso_init(const SwarmArgs& a, int sms, cudaStream_t st);
void launch_pso_move(const SwarmArgs& a, int sms, cudaStream_t st);
void launch_de_trial(const SwarmArgs& a, int sms, cudaStream_t st);
void launch_da_start(const SwarmArgs& a, int sms, cudaStream_t st);
void launch_da_visit(const SwarmArgs& a, int j, int sms, cudaStream_t st);
void launch_da_accept(const SwarmArgs& a, const double* cost, int j, int sms, cudaStream_t st);
void launch_da_best(const SwarmArgs& a, int sms, cudaStream_t st);
void launch_pso_best(const SwarmArgs& a, const double* cost, int sms, cudaStream_t st);
// Bests of the generation just evaluated and (move) the positions of the next one, for
// populations of at most PSO_STEP_MAX_P.
constexpr int PSO_STEP_MAX_P = 1024;
// Whether a batch's generations take it, or k_pso_best and k_pso_move: it has one block per
// spectrum, so with few spectra a population of many coordinates (particles x poles) leaves
// the GPU idle, where the move of its own spreads over it. Whole fits, separate kernels
// against one, ms: 1 spectrum, 100 generations, 64 particles x 3 poles 2.08 and 1.87, 128 x
// 10 3.85 and 3.85, 256 x 10 3.90 and 4.29, 1024 x 20 7.75 and 13.15; 64 spectra, 128 x 10
// 12.37 and 12.18, 200 x 10 (60 generations) 8.02 and 8.01, 512 x 10 21.8 and 22.4; 152
// spectra, 256 x 20 53.3 and 53.3, 1024 x 20 92.4 and 97.6; 1024 spectra, 256 x 12 (60)
// 26.8 and 25.9, 1024 x 20 (60) 365 and 356.
inline bool pso_step_fused(int64_t S, int P, int n_max) {
  const int64_t coords = (int64_t)P * n_max;   // k_pso_move's blocks take 16 particles, 256 coordinates at a time
  return P <= PSO_STEP_MAX_P && (coords <= (n_max > 16 ? 1536 : 1280) || coords <= 32 * S);
}
void launch_pso_step(const SwarmArgs& a, const double* cost, bool move, int sms, cudaStream_t st);
// Step lengths of a polish line evaluated in a round, and whether one round takes all
// `trials` of them (at most 32). Its launches are saved then (one spectrum, 8 lines: 7 per
// iteration), but a line that rejects every step evaluates all of them at once, so the GPU
// has to have room: at most 256 trials per SM over all lines, and fewer where one costs more
// (poles; FP64; without tables, samples). Whole fits, rounds against one round, ms, 8 lines
// per spectrum, 19 step lengths (the default): mixed, 1 spectrum, 3 poles 3.62 and 3.08; 64,
// 8 poles 7.99 and 6.43; 128, 20 poles of 4000 samples 38.7 and 38.2; 192, 8 poles of 1000
// 7.83 and 7.43, of 4000 17.4 and 17.8; 256, 4 poles 3.48 and 3.03, 8 poles of 1000 8.66 and
// 8.70, 12 12.6 and 13.3, 20 21.4 and 24.0. Tables, 256, 12 poles 4.83 and 4.55, 20 poles 7.76
// and 8.06. FP64 column sums, 64, 20 poles of 400 samples 104 and 96; 128, 12 poles 68.0 and
// 68.6, 20 poles 135 and 140; 256, 4 poles 30.2 and 29.2, 8 poles 64.2 and 67.2.
constexpr int POLISH_R = 8;
inline bool polish_one_round(int64_t lines, int trials, int n_max, int64_t longest, int precision, int sms) {
  if (trials <= POLISH_R || trials > 32 || lines * trials > 256 * (int64_t)sms) return false;
  const double per_sm = (double)(lines * trials) / sms, work = per_sm * (n_max + 8);
  if (precision == DEBYE_PREC_MIXED_TABLE) return work <= 5750.0;
  if (precision == DEBYE_PREC_MIXED) return work <= 3000.0 || work * (double)(longest + 4000) <= 20.5e6;
  return per_sm * (n_max + 2) <= 1800.0;
}
void launch_gen_advance(int* gen, cudaStream_t st);
void launch_add_scalar(double* dst, double v, cudaStream_t st);
void launch_topk(const SwarmArgs& a, const PolishArgs& pa, int sms, cudaStream_t st);
void launch_polish_start(const PolishArgs& pa, int sms, cudaStream_t st);
void launch_polish_take0(const PolishArgs& pa, int sms, cudaStream_t st);
void launch_polish_step(const PolishArgs& pa, const int32_t* n_poles, const double* lo, const double* hi,
                        int sms, cudaStream_t st);
void launch_polish_first(const PolishArgs& pa, const int32_t* n_poles, const double* lo, const double* hi,
                         const int64_t* offsets, int sms, cudaStream_t st);
void launch_polish_accept(const PolishArgs& pa, const int32_t* n_poles, const double* lo, const double* hi,
                          const int64_t* offsets, int sms, cudaStream_t st);
void launch_polish_take(const PolishArgs& pa, const int32_t* n_poles, int sms, cudaStream_t st);
void launch_pick_best(const SwarmArgs& a, const PolishArgs& pa, double* out_theta, int sms, cudaStream_t st);
void launch_assemble(int64_t S, int nmax, const int32_t* n_poles, const double* theta, const double* weights,
                     const double* cost, double* eps_inf, double* d_eps, double* tau, double* final_cost,
                     int sms, cudaStream_t st);

}  // namespace debyefit
