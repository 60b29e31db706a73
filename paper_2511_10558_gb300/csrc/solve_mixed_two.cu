// Instantiations of the solver kernels (BDF and ESDIRK), LT = float, matrix in shared memory, two cells on an SM.
#define CBX_THREADS 256
#define CBX_CTAS 2
#define CBX_MAX_S 160
#define CBX_LEAN 1
#include "solver_dev.cuh"

namespace cbx {

int launch_solve_mixed_two(const SolveArgs& a, bool rk, size_t smem, int grid, void* stream) {
  return rk ? launch_t<float, false, true>(a, smem, grid, (cudaStream_t)stream)
            : launch_t<float, false>(a, smem, grid, (cudaStream_t)stream);
}

int occupancy_solve_mixed_two(size_t smem) { return occupancy_t<float, false>(smem); }

}  // namespace cbx
