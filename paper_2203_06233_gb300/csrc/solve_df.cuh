// The double-float weight solve (solve_df.cu): parameters and launcher.
#pragma once

#include <type_traits>

#include "stap_internal.cuh"

namespace stap {

// Largest bound D / load_factor + 1 on the loaded matrix's condition number
// at which the double-float kernels stand in for the FP64 ones.
constexpr double kDfMaxKappa = 524288.0;   // 2^19

// Whether a plan's solve takes these kernels: the refinement option, and the
// default solver where the load bounds the condition number.
inline bool solve_df_eligible(int solver, double load_factor, int D) {
  return solver == STAP_SOLVE_MIXED_IR ||
         (load_factor > 0.0 && (double)D / load_factor + 1.0 <= kDfMaxKappa);
}

// Parameters of one launch (one CPI); gx = the launch's grid size.
struct SolveDfParams {
  const double2* cov;      // [nsys][D][D], lower triangle and real diagonal read
  float2* wts;             // [nsys][S][D]
  const float4* steer_ff;  // [S][D] steering vectors (re hi, re lo, im hi, im lo)
  const float4* g_ff;      // [T] temporal factors (separable steering)
  const float4* sep_a_ff;  // [S][C] spatial factors (separable steering)
  long long nsys;
  int D, S, C;
  int sep;                 // solve the C basis right-hand sides g (x) e_c
  int sym;                 // separable factors with a_{S-1-s} = conj(a_s)
  double load_factor;
  int refine_steps;
  DeviceStatus* status;
  int gx;
};

// D <= 32 and D > 32, double-float throughout; and with the FP32 factor and
// substitutions of STAP_SOLVE_MIXED_IR (double-float residuals and solutions).
// One translation unit each.
cudaError_t launch_solve_df_small(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_big(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_small_ir(const SolveDfParams& p, cudaStream_t s);
cudaError_t launch_solve_df_big_ir(const SolveDfParams& p, cudaStream_t s);

cudaError_t check_record_solve_df_small(CheckRecord* out);
cudaError_t check_record_solve_df_big(CheckRecord* out);
cudaError_t check_record_solve_df_small_ir(CheckRecord* out);
cudaError_t check_record_solve_df_big_ir(CheckRecord* out);

}  // namespace stap
