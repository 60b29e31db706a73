// Launch planning of the solver kernel (host code): shared-memory and
// workspace sizes, the matrix placement, occupancy, and the dispatch to the
// translation unit holding each kernel instantiation.
#include "solver_dev.cuh"

namespace cbx {

size_t smem_bytes(int S, int R, int nseg, bool mixed, bool gm, int piv_ints) {
  return layout(S, R, nseg, mixed, gm, nullptr, nullptr, piv_ints);
}

long long workspace_doubles(int S, int R, int nnzJ, bool mixed, bool gm) {
  long long n = 3LL * R + nnzJ;
  n = (n + 31) / 32 * 32;
  if (gm) n += ((long long)S * lead_dim_gm(S) * (mixed ? 4 : 8) / 8 + 31) / 32 * 32;
  return n;
}

namespace {

// Shared memory of an SM, and what each resident CTA takes of it beside its
// dynamic part (1 KB reserved by the system, the kernel's static variables).
constexpr size_t kSmShared = 228 * 1024, kCtaReserved = 1024 + 128;

struct ShapeKernel {
  int (*launch)(const SolveArgs&, bool rk, size_t smem, int grid, void* stream);
  int (*occupancy)(size_t smem);
};

// The kernel of a plan with several CTAs per SM.
ShapeKernel shape_kernel(const SolverPlan& p) {
  if (p.gm)
    return p.mixed ? ShapeKernel{launch_solve_mixed_gm_two, occupancy_solve_mixed_gm_two}
                   : ShapeKernel{launch_solve_fp64_gm_two, occupancy_solve_fp64_gm_two};
  if (p.shape == kNarrow)
    return p.mixed ? ShapeKernel{launch_solve_mixed_narrow, occupancy_solve_mixed_narrow}
                   : ShapeKernel{launch_solve_fp64_narrow, occupancy_solve_fp64_narrow};
  if (p.shape == kMid)
    return p.mixed ? ShapeKernel{launch_solve_mixed_mid, occupancy_solve_mixed_mid}
                   : ShapeKernel{launch_solve_fp64_mid, occupancy_solve_fp64_mid};
  return p.mixed ? ShapeKernel{launch_solve_mixed_two, occupancy_solve_mixed_two}
                 : ShapeKernel{launch_solve_fp64_two, occupancy_solve_fp64_two};
}

}  // namespace

SolverPlan plan_solver(int S, int R, int nseg, int nnzJ, bool mixed, int head_ints, int C) {
  SolverPlan p;
  p.mixed = mixed;
  const size_t optin = device_smem_optin() - kStaticShared;
  // shared-memory matrix when it fits and the FP64 LU's register tiling allows (S <= 256)
  p.gm = !(S <= 32 * kMaxColRegs && smem_bytes(S, R, nseg, mixed, false) <= optin);
  p.smem = smem_bytes(S, R, nseg, mixed, p.gm);
  // FP64 shared-memory solver: stage the sparse pivots' lists when they fit
  if (!mixed && !p.gm && smem_bytes(S, R, nseg, false, false, head_ints) <= optin) {
    p.piv_ints = head_ints;
    p.smem = smem_bytes(S, R, nseg, false, false, head_ints);
  }
  p.ws_stride = workspace_doubles(S, R, nnzJ, mixed, p.gm);
  p.occupancy = 0;
  if (S > 2 * NT || p.smem > optin) return p;
  if (mixed)
    p.occupancy = p.gm ? occupancy_solve_mixed_gm(p.smem) : occupancy_solve_mixed(p.smem);
  else
    p.occupancy = p.gm ? occupancy_solve_fp64_gm(p.smem) : occupancy_solve_fp64(p.smem);
  if (p.occupancy < 1) return p;
  // Batches: several cells per SM. A cell is slower beside others (they share
  // the FP64 pipe) but leaves the SM fewer idle cycles, so a shape pays once the
  // batch is bound by throughput rather than by its costliest cell; the more
  // of a cell's time is serial (small networks), the sooner. Measured with
  // cells of 1e5 yr (500 species: 1e3 yr), times in ms by cells:
  //   32 species:  160/304/608/1216 cells, one per SM 17/24/41/77, mid
  //                13/13/16/30, narrow 15/14/16/22
  //   61:          one 57/67/127/227, two 60/64/95/163, mid 64/66/72/125
  //   80:          one 39/58/93/169, two 37/51/70/117, mid 40/57/67/102
  //   97:          one 92/80/121/224, two 99/92/93/167 (mixed, 304/608/1216:
  //                one 77/115/215, two 83/84/148)
  //   150 mixed:   one 81/84/86/174, two 92/104/119/130
  //   500 mixed:   160/304/608 cells, one 137/210/365, two 150/181/292;
  //   500 FP64:    304 cells, one 743, two 647; 200 FP64: 304/608 cells, one
  //                210/355, two 214/270
  const double load = (double)C / device_sm_count();  // cells per SM
  const bool lean_ok = nseg <= R;
  const size_t full = p.smem, lean = layout(S, R, nseg, mixed, p.gm, nullptr, nullptr, 0, true);
  auto fits = [&](size_t smem, int ctas) { return (smem + kCtaReserved) * ctas <= kSmShared; };
  CtaShape shape = kOnePerSm;
  if (p.gm) {
    if (load >= (S > 256 ? 2.0 : 4.0) && lean_ok && fits(lean, 2)) shape = kTwoPerSm;
  } else if (S <= 48 && load >= 6.0 && fits(full, 5)) {
    shape = kNarrow;
  } else if (S <= 96 && load > (S <= 48 ? 1.0 : 4.0) && lean_ok && fits(lean, 3)) {
    shape = kMid;
  } else if (S <= (mixed ? 160 : 128) && load >= (S <= 96 ? 1.5 : mixed && S > 112 ? 6.0 : 4.0) && lean_ok &&
             fits(lean, 2)) {
    shape = kTwoPerSm;
  }
  if (shape == kOnePerSm) return p;
  SolverPlan b = p;
  b.shape = shape;
  if (shape != kNarrow) {
    b.smem = lean;
    b.piv_ints = 0;
  }
  b.occupancy = shape_kernel(b).occupancy(b.smem);
  return b.occupancy > p.occupancy ? b : p;
}

int launch_solver(const SolveArgs& a0, const SolverPlan& p, int grid, void* stream) {
  SolveArgs a = a0;
  a.piv_ints = p.piv_ints;
  if (p.shape != kOnePerSm) return shape_kernel(p).launch(a, false, p.smem, grid, stream);
  if (p.mixed)
    return p.gm ? launch_solve_mixed_gm(a, p.smem, grid, stream) : launch_solve_mixed(a, p.smem, grid, stream);
  return p.gm ? launch_solve_fp64_gm(a, p.smem, grid, stream) : launch_solve_fp64(a, p.smem, grid, stream);
}

int device_sm_count() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  return v;
}

size_t device_smem_optin() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return (size_t)v;
}

int launch_solver_rk(const SolveArgs& a0, const SolverPlan& p, int grid, void* stream) {
  SolveArgs a = a0;
  a.piv_ints = p.piv_ints;
  if (p.shape != kOnePerSm) return shape_kernel(p).launch(a, true, p.smem, grid, stream);
  if (p.gm)
    return p.mixed ? launch_solve_mixed_gm_rk(a, p.smem, grid, stream) : launch_solve_fp64_gm_rk(a, p.smem, grid, stream);
  return p.mixed ? launch_solve_mixed_rk(a, p.smem, grid, stream) : launch_solve_fp64_rk(a, p.smem, grid, stream);
}

}  // namespace cbx
