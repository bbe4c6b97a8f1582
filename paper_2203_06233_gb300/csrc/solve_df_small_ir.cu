// The double-float weight solve (solve_df_kernel.cuh) for D <= 32: FP32 factor and substitutions.
#include "solve_df_kernel.cuh"

namespace stap {

cudaError_t launch_solve_df_small_ir(const SolveDfParams& p, cudaStream_t s) {
  const int D = p.D;
  if (D <= 8) return launch_df<4, 2, 16, true>(p, s);
  if (D <= 12) return launch_df<4, 3, 16, true>(p, s);
  if (D <= 16) return launch_df<4, 4, 16, true>(p, s);
  if (D <= 24) return launch_df<8, 3, 64, true>(p, s);
  return launch_df<8, 4, 64, true>(p, s);
}

cudaError_t check_record_solve_df_small_ir(CheckRecord* out) { return read_check_record(out); }

}  // namespace stap
