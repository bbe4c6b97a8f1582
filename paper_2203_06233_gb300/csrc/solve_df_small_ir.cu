// The double-float weight solve (solve_df_kernel.cuh) for D <= 32: FP32 factor and substitutions.
#include "solve_df_kernel.cuh"

namespace stap {

cudaError_t launch_solve_df_small_ir(const SolveDfParams& p, cudaStream_t s) {
  const int D = p.D;
  // launch_small's splits.  128 threads per system where there are few
  // (us, without / with: D = 13 C = 13 S = 16, 128 systems 53 / 22, 512 53 / 31;
  // D = 15 C = 5, 512 systems 35 / 27, 1024 39 / 53; D = 20 C = 20 S = 64, 128 systems
  // 107 / 67, 512 120 / 92, 1024 171 / 171)
  const int nrhs = p.sep ? p.C : p.S;
  const bool few = p.cpi_sys <= 512, many = nrhs > 4 || p.S > 16;
  if (D <= 8) return many && few ? launch_df<4, 2, 128, kMixedIr>(p, s) : launch_df<4, 2, 16, kMixedIr>(p, s);
  if (D <= 12 && p.cpi_sys >= 2048) return launch_df<4, 3, 16, kMixedIr>(p, s);
  if (D <= 16) return many && few ? launch_df<8, 2, 128, kMixedIr>(p, s) : launch_df<8, 2, 32, kMixedIr>(p, s);
  if (D <= 24) return nrhs > 8 && few ? launch_df<8, 3, 128, kMixedIr>(p, s) : launch_df<8, 3, 64, kMixedIr>(p, s);
  return launch_df<16, 2, 128, kMixedIr>(p, s);
}

cudaError_t check_record_solve_df_small_ir(CheckRecord* out) { return read_check_record(out); }

}  // namespace stap
