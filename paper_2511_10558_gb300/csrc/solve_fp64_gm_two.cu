// Instantiations of the solver kernels (BDF and ESDIRK), LT = double, matrix in the CTA's global workspace, two
// cells on an SM.
#define CBX_THREADS 256
#define CBX_CTAS 2
#define CBX_LEAN 1
#include "solver_dev.cuh"

namespace cbx {

int launch_solve_fp64_gm_two(const SolveArgs& a, bool rk, size_t smem, int grid, void* stream) {
  return rk ? launch_t<double, true, true>(a, smem, grid, (cudaStream_t)stream)
            : launch_t<double, true>(a, smem, grid, (cudaStream_t)stream);
}

int occupancy_solve_fp64_gm_two(size_t smem) { return occupancy_t<double, true>(smem); }

}  // namespace cbx
