// Launch planning of the solver kernel (host code): shared-memory and
// workspace sizes, the matrix placement, occupancy, and the dispatch to the
// translation unit holding each kernel instantiation.
#include <algorithm>

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

// Whether the network can take a shape with several CTAs on an SM: the most
// species that its kernels hold, and the shared memory of its CTAs.
bool takes(const LaunchForms& f, CtaShape shape) {
  const SolverPlan& one = f.form[kOnePerSm];
  auto fits = [&](size_t smem, int ctas) { return (smem + kCtaReserved) * ctas <= kSmShared; };
  if (shape == kNarrow) return !one.gm && f.S <= 48 && fits(one.smem, 5);
  if (f.nseg > f.R) return false;  // no room for the segment sums in the lean layout
  if (shape == kMid) return !one.gm && f.S <= 96 && fits(f.lean, 3);
  return (one.gm || f.S <= (one.mixed ? 160 : 128)) && fits(f.lean, 2);
}

// Batches: several cells per SM. A cell is slower beside others (they share
// the FP64 pipe) but leaves the SM fewer idle cycles, so a shape pays once the
// batch is bound by throughput rather than by its costliest cell; the more
// of a cell's time is serial (small networks), the sooner. Measured on one GB300
// (152 SMs), ms, medians of five calls (which differ by 2 to 10 %, by up to 20 %
// where few cells end a launch), by cells; BDF, 32 to 80 species 1e5 yr, 96 to
// 200 1e4, 500 1e3:
//               cells      153   200   304   456   608   912  1216  2432
//   32 FP64     one         14    20    24          42    59    77   144
//               mid         13    13    14          16    25    30    52
//               narrow      14    14    15          16    19    22    42
//   48 FP64     one         15    19    23          41    58    76   147
//               mid         17    16    18          22    30    36    66
//               narrow      23    22    24          26    33    39    63
//   61 FP64     one         53    66    68    98   126   157   210
//               two         56    60    58    77    92   117   149
//               mid         62    61    62    68    78   103   123
//   80 mixed    one         36          62    84   103   147   191
//               two         36          47    60    75   102   130
//               mid         37          47    59    67    86   111
//   96 FP64     one         33          44    58    71   100   130
//               two         35          48    53    56    74    95
//   97 FP64     one         35          58    69    89   128   167
//               two         37          67    56    67    93   120
//   150 mixed   one         53          60          64    79   105 (1501: 131)
//               two         62          75          90    89    86 (1501: 100)
//   200 FP64    one        143         182   254   327
//               two        151         219   241   277
//   500 mixed   one         95         153   212   269
//               two        113         148   180   227
//   500 FP64    one        442         696   929
//               two        479         663   860
// The line moves with the span, as the costliest cells' share does: 150 mixed, 912
// cells over 1e2 and 1e6 yr, one 48 and 175, two 37 and 146; 500 mixed, 304 cells
// over 1e4 yr, one 218, two 268. The ESDIRK's solves are more of its time, which
// moves it too; just above one cell an SM, at 45 to 48 species, mid was slower
// with it than one to an SM (153 cells of 48: 53 against 49 ms; 160: 41 against
// 38), so mid begins there at 1.1.
CtaShape batch_shape(const LaunchForms& f, int C) {
  const SolverPlan& one = f.form[kOnePerSm];
  const double load = (double)C / one.sms;  // cells per SM
  if (one.gm) return load >= (f.S > 256 ? 2.0 : 4.0) && takes(f, kTwoPerSm) ? kTwoPerSm : kOnePerSm;
  if (load >= 6.0 && takes(f, kNarrow)) return kNarrow;
  if (load > (f.S <= 44 ? 1.0 : f.S <= 48 ? 1.1 : 4.0) && takes(f, kMid)) return kMid;
  if (load >= (f.S <= 96 ? 1.5 : one.mixed && f.S > 112 ? 6.0 : 4.0) && takes(f, kTwoPerSm)) return kTwoPerSm;
  return kOnePerSm;
}

// The plan of a shape with several CTAs on an SM, or that of one cell to an SM
// where the device would not run more CTAs of it.
void query_form(LaunchForms& f, CtaShape shape) {
  const SolverPlan& one = f.form[kOnePerSm];
  SolverPlan p = one;
  p.shape = shape;
  if (shape != kNarrow) {
    p.smem = f.lean;
    p.piv_ints = 0;
  }
  p.occupancy = shape_kernel(p).occupancy(p.smem);
  f.form[shape] = p.occupancy > one.occupancy ? p : one;
}

LaunchForms base_form(int S, int R, int nseg, int nnzJ, bool mixed, int head_ints) {
  LaunchForms f;
  f.S = S;
  f.R = R;
  f.nseg = nseg;
  SolverPlan& p = f.form[kOnePerSm];
  p.mixed = mixed;
  p.sms = device_sm_count();
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
  if (S > 2 * NT || p.smem > optin) return f;
  if (mixed)
    p.occupancy = p.gm ? occupancy_solve_mixed_gm(p.smem) : occupancy_solve_mixed(p.smem);
  else
    p.occupancy = p.gm ? occupancy_solve_fp64_gm(p.smem) : occupancy_solve_fp64(p.smem);
  f.lean = layout(S, R, nseg, mixed, p.gm, nullptr, nullptr, 0, true);
  return f;
}

template <typename Form>
SolverPlan choose(const LaunchForms& f, int C, const LaunchLimits& limits, Form form) {
  const SolverPlan& one = f.form[kOnePerSm];
  const int ctas = limits.max_ctas;
  if (ctas > 0 && ctas <= one.sms) return one;
  // (Under a cap on SMs too the cells count against the whole device, which other
  // launches share: against the capped SMs a server's requests took 8.70 s, so
  // 8.44; small bursts 17.4 and 16.7 ms.)
  const SolverPlan p = form(batch_shape(f, C));
  // A limit that leaves less than half of the shape's CTAs: the shape for as many
  // cells as it lets run at a time (48 species, 150 CTAs: narrow 23 ms, one to an
  // SM 15; 150 species mixed, 204 of 304 CTAs: two to an SM 126, one 130).
  return ctas > 0 && ctas < std::min(C, p.occupancy * one.sms) / 2 ? form(batch_shape(f, ctas)) : p;
}

}  // namespace

LaunchForms launch_forms(int S, int R, int nseg, int nnzJ, bool mixed, int head_ints) {
  LaunchForms f = base_form(S, R, nseg, nnzJ, mixed, head_ints);
  if (f.form[kOnePerSm].occupancy < 1) return f;
  for (CtaShape shape : {kNarrow, kMid, kTwoPerSm})
    if (takes(f, shape)) query_form(f, shape);
  return f;
}

SolverPlan choose_form(const LaunchForms& f, int C, const LaunchLimits& limits) {
  return choose(f, C, limits, [&](CtaShape s) { return f.form[s]; });
}

SolverPlan plan_solver(int S, int R, int nseg, int nnzJ, bool mixed, int head_ints, int C,
                       const LaunchLimits& limits) {
  LaunchForms f = base_form(S, R, nseg, nnzJ, mixed, head_ints);
  if (f.form[kOnePerSm].occupancy < 1) return f.form[kOnePerSm];
  return choose(f, C, limits, [&](CtaShape s) {
    if (s != kOnePerSm) query_form(f, s);
    return f.form[s];
  });
}

int launch_grid(const SolverPlan& p, int C, const LaunchLimits& limits) {
  const int sms = limits.max_sms > 0 ? std::min(limits.max_sms, p.sms) : p.sms;
  const int grid = std::min(C, p.occupancy * sms);
  return limits.max_ctas > 0 ? std::min(grid, limits.max_ctas) : grid;
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
