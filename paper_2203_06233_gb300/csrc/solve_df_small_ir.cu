// The double-float weight solve (solve_df_kernel.cuh) for D <= 32: FP32 factor and substitutions.
#include "solve_df_kernel.cuh"

namespace stap {

cudaError_t launch_solve_df_small_ir(const SolveDfParams& p, cudaStream_t s) {
  const int D = p.D;
  // D <= 12: half a warp per system, or a whole one where the systems are too
  // few to fill the SMs and the latency of one counts (C 4 S 16, D = 12, half /
  // whole: 256 systems 34.4 / 26.3 us, 1024 36.5 / 30.3, 4096 58.0 / 65.9).  D = 16:
  // a warp (1024: half 55.5, whole 36.4; 16384: 299, 277).  D = 32: 128 threads
  // (256: 64 threads 82.1, 128 58.0; 16384: 1875, 1817)
  if (D <= 8 || (D <= 12 && p.cpi_sys >= 2048))
    return D <= 8 ? launch_df<4, 2, 16, kMixedIr>(p, s) : launch_df<4, 3, 16, kMixedIr>(p, s);
  if (D <= 16) return launch_df<8, 2, 32, kMixedIr>(p, s);
  if (D <= 24) return launch_df<8, 3, 64, kMixedIr>(p, s);
  return launch_df<16, 2, 128, kMixedIr>(p, s);
}

cudaError_t check_record_solve_df_small_ir(CheckRecord* out) { return read_check_record(out); }

}  // namespace stap
