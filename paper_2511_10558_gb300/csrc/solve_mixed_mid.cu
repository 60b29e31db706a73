// Instantiations of the solver kernels (BDF and ESDIRK), LT = float, matrix in shared memory: 128 threads a cell,
// up to 96 species, three or four cells on an SM.
#define CBX_THREADS 128
#define CBX_CTAS 4
#define CBX_MAX_S 96
#define CBX_LEAN 1
#include "solver_dev.cuh"

namespace cbx {

int launch_solve_mixed_mid(const SolveArgs& a, bool rk, size_t smem, int grid, void* stream) {
  return rk ? launch_t<float, false, true>(a, smem, grid, (cudaStream_t)stream)
            : launch_t<float, false>(a, smem, grid, (cudaStream_t)stream);
}

int occupancy_solve_mixed_mid(size_t smem) { return occupancy_t<float, false>(smem); }

}  // namespace cbx
