// Instantiations of the solver kernels (BDF and ESDIRK), LT = double, matrix in shared memory: 64 threads a cell,
// up to 64 species, up to eight cells on an SM.
#define CBX_THREADS 64
#define CBX_CTAS 8
#define CBX_MAX_S 64
#include "solver_dev.cuh"

namespace cbx {

int launch_solve_fp64_narrow(const SolveArgs& a, bool rk, size_t smem, int grid, void* stream) {
  return rk ? launch_t<double, false, true>(a, smem, grid, (cudaStream_t)stream)
            : launch_t<double, false>(a, smem, grid, (cudaStream_t)stream);
}

int occupancy_solve_fp64_narrow(size_t smem) { return occupancy_t<double, false>(smem); }

}  // namespace cbx
