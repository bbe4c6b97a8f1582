// The double-float weight solve (solve_df_kernel.cuh) for D > 32: FP32 factor and substitutions.
#include "solve_df_kernel.cuh"

namespace stap {

cudaError_t launch_solve_df_big_ir(const SolveDfParams& p, cudaStream_t s) {
  const int D = p.D;
  if (D <= 48) return launch_df<16, 3, 256, kMixedIr>(p, s);
  if (D <= 64) return launch_df<16, 4, 256, kMixedIr>(p, s);
  if (D <= 96) return launch_df<16, 6, 512, kMixedIr>(p, s);
  return launch_df<16, 8, 512, kMixedIr>(p, s);
}

cudaError_t check_record_solve_df_big_ir(CheckRecord* out) { return read_check_record(out); }

}  // namespace stap
