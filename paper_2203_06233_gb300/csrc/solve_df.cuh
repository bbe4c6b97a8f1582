// The double-float weight solve (solve_df_kernel.cuh): parameters and launchers.
#pragma once

#include <type_traits>

#include "stap_internal.cuh"

namespace stap {

// Largest bound D / load_factor + 1 on the loaded matrix's condition number
// at which the double-float kernels stand in for the FP64 ones.  What it
// guarantees: for R positive semidefinite, as a sample covariance is, kappa(Rl)
// is at most this and each weight vector is off by less than its complex64
// rounding, whether it was solved by itself or combined from the basis
// solutions (those whose combination cancels are solved by themselves).  For
// any other Hermitian R, as a caller may pass one, nothing bounds kappa:
// the kernels for any matrix then look at what the first refinement step corrects.
constexpr double kDfMaxKappa = 524288.0;   // 2^19

// A system that the kernels for any matrix cannot answer for has this in
// the first word of its weights until the FP64 kernel has solved it: a NaN that
// no arithmetic gives.
constexpr unsigned kUnsolved = 0x7FD5A3E1u;

// Whether a plan's solve takes these kernels: the refinement option, and the
// default solver where the load bounds the condition number.  Without a
// refinement step, on grids (D > 32), the bound is a quarter of that: a vector
// along strong interference loses up to kappa 2^-42 (measured at D = 128: 3e-7 at
// kappa 2^19, 8e-8 at 2^17).  One or two rows are left to FP64, a lane of which
// does a whole right-hand side (D = 1, 16384 systems, S = 2: 6.6 us, in
// double-float 21.6).
inline bool solve_df_eligible(int solver, double load_factor, int D, int refine_steps) {
  const double most = refine_steps == 0 && D > kSmallMaxD ? kDfMaxKappa / 4 : kDfMaxKappa;
  return solver == STAP_SOLVE_MIXED_IR ||
         (load_factor > 0.0 && (double)D / load_factor + 1.0 <= most && D > 2);
}

// Parameters of one launch (one CPI); gx = the launch's grid size.
struct SolveDfParams {
  const double2* cov;      // [nsys][D][D], lower triangle and real diagonal read
  float2* wts;             // [nsys][S][D]
  const float4* steer_ff;  // [S][D] steering vectors (re hi, re lo, im hi, im lo)
  const float4* g_ff;      // [T] temporal factors (separable steering)
  const float4* sep_a_ff;  // [S][C] spatial factors (separable steering)
  // separable steering: a u_s whose largest entry is below `cancel` times the
  // sum of the basis solutions' largest needs a solve of its own; one with q =
  // Re v^H u of cancel_q / delta or more cannot be
  float cancel, cancel_q;
  float steer_sum;         // the largest sum of |re| + |im| over a steering vector
  long long nsys;
  long long cpi_sys;       // of the whole CPI: a launch may cover a range slab of it.  Where
                           // kernels round differently this one chooses, so that slabs agree
  int D, S, C;
  int sep;                 // solve the C basis right-hand sides g (x) e_c
  int sym;                 // separable factors with a_{S-1-s} = conj(a_s)
  double load_factor;
  int refine_steps;
  float max_correction;    // any matrix: systems that fail, or whose first correction is above
                           // this part of the solution, are marked instead of counted
  DeviceStatus* status;
  int gx;
};

// D <= 32 and D > 32: double-float throughout, of covariances and of any
// Hermitian matrices; and with the FP32 factor and substitutions of
// STAP_SOLVE_MIXED_IR (double-float residuals and solutions).  One translation
// unit each.
cudaError_t launch_solve_df_small(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_big(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_small_any(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_big_any(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_small_ir(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_big_ir(const SolveDfParams& p, cudaStream_t s);

cudaError_t check_record_solve_df_small(CheckRecord* out);
cudaError_t check_record_solve_df_big(CheckRecord* out);
cudaError_t check_record_solve_df_small_any(CheckRecord* out);
cudaError_t check_record_solve_df_big_any(CheckRecord* out);
cudaError_t check_record_solve_df_small_ir(CheckRecord* out);
cudaError_t check_record_solve_df_big_ir(CheckRecord* out);

}  // namespace stap
