// The double-float weight solve (solve_df_kernel.cuh) for D > 32: double-float throughout, of any Hermitian matrix.
#include "solve_df_kernel.cuh"

namespace stap {

cudaError_t launch_solve_df_big_any(const SolveDfParams& p, cudaStream_t s) { return launch_large<kAnyMatrix>(p, s); }

cudaError_t check_record_solve_df_big_any(CheckRecord* out) { return read_check_record(out); }

}  // namespace stap
