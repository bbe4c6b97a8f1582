// The double-float weight solve (solve_df_kernel.cuh) for D > 32: double-float throughout.
#include "solve_df_kernel.cuh"

namespace stap {

cudaError_t launch_solve_df_big(const SolveDfParams& p, cudaStream_t s) {
  const int D = p.D;
  if (D <= 48) return launch_df<16, 3, 256, false>(p, s);
  if (D <= 64) return launch_df<16, 4, 256, false>(p, s);
  if (D <= 96) return launch_df<16, 6, 512, false>(p, s);
  return launch_df<32, 4, 512, false>(p, s);
}

cudaError_t check_record_solve_df_big(CheckRecord* out) { return read_check_record(out); }

}  // namespace stap
