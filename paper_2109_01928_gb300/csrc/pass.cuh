// Launch of the pass kernels of one pole count N (included by pass_b*.cu).
#pragma once
#include "eval.cuh"
#include "launch.h"
#include "solve_sums.cuh"

namespace debyefit {

// The column-sum passes (PH_SUMS, PH_SUMSG) and the per-N column-sum solves
// (PH_SOLVE, PH_SOLVEG) are the mixed-precision path; the
// Gram, residual and gradient passes the FP64 path.
template <int N>
void launch_pass_n(int phase, const EvalArgs& a, int grid, int block, cudaStream_t st) {
  // the column-sum pass sweeps at most SQUARED_CHUNK poles at a time, which fits 168
  // registers (3 resident 128-thread blocks; 4 blocks, 128 registers: N = 12 1.109 ms
  // against 1.065 ms); with the derivative sums 2 blocks
  constexpr int MB_SUMS = 3, MB_SUMSG = 2;
  constexpr int MAXT = N <= 12 ? 128 : 256;
  switch (phase) {
    case PH_SUMS: k_pass_sums<N, false, MAX_BLOCK, MB_SUMS><<<grid, block, 0, st>>>(a); break;
    case PH_SUMSG: k_pass_sums<N, true, MAX_BLOCK, MB_SUMSG><<<grid, block, 0, st>>>(a); break;
    case PH_GRAM: k_pass<PH_GRAM, N, N, MAXT, 1><<<grid, block, 0, st>>>(a); break;
    case PH_GRAM_SUMS: k_pass<PH_GRAM_SUMS, N, N, MAXT, 1><<<grid, block, 0, st>>>(a); break;
    case PH_REFINE: k_pass<PH_REFINE, N, N, MAXT, 1><<<grid, block, 0, st>>>(a); break;
    case PH_SOLVE:
    case PH_SOLVEG:
      if constexpr (N >= SOLVE_ROLL_FROM) {   // a warp per block: `block` candidates per unit in slices of 32
        const int slices = block / 32, g = std::min(grid, a.n_units) * slices;
        const void* k = phase == PH_SOLVE ? (const void*)k_solve_rows<N, 0> : (const void*)k_solve_rows<N, 1>;
        if constexpr (solve_roll_bytes(N) > 48 * 1024)   // set with every launch: the attribute goes with the context
          cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)solve_roll_bytes(N));
        if (phase == PH_SOLVE)
          k_solve_rows<N, 0><<<g, 32, solve_roll_bytes(N), st>>>(a, slices, a.out_cost, a.out_weights, nullptr);
        else
          k_solve_rows<N, 1><<<g, 32, solve_roll_bytes(N), st>>>(a, slices, a.out_cost, a.out_weights, a.out_grad);
      } else if (phase == PH_SOLVE) {         // one thread per candidate
        k_solve_sums_t<N, 0><<<grid, block, 0, st>>>(a, a.out_cost, a.out_weights, nullptr);
      } else {
        k_solve_sums_t<N, 1><<<grid, block, 0, st>>>(a, a.out_cost, a.out_weights, a.out_grad);
      }
      break;
    default: k_pass<PH_GRAD, N, N, MAXT, 1><<<grid, block, 0, st>>>(a); break;
  }
}

}  // namespace debyefit
