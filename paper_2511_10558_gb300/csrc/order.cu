// The order in which a launch's persistent CTAs take its cells: costly first.
//
// A batch ends when its slowest CTA does. Cells differ in cost by a factor of
// 6 to 10 (irradiated gas goes on evolving, shielded gas reaches its steady
// state), so taking them in the caller's order leaves one CTA working on a
// costly cell that it took last while the others idle: 150 species, FP64,
// 1,216 cells to 1e4 yr took 232 ms of which 171 ms were work. With the costly
// cells first the tail is filled by cheap ones. Results do not depend on the
// order (a cell's arithmetic is the same on any CTA).
//
// The estimate of a solve is the number of photo-reaction and cosmic-ray times
// in the cell's span, (alpha_ph G0 exp(-gamma_ph A_V) + alpha_cr zeta)(t_end -
// t0) with the network's mean parameters: measured on 150 species, the mean
// cost is monotone in it (A_V deciles, 1 Myr: 129, 102, 63 and then 26 ms a
// cell). The reverse sweep's cost is known: the ops on the tape. Cells are
// sorted into 256 logarithmic buckets by one CTA: two passes over the inputs
// (a few microseconds, bound by latency; C up to a few thousand is one or two
// loads a thread), so it is launched only when a CTA has to take more than one
// cell.
#include <cuda_runtime.h>

#include <cmath>

#include "internal.h"

namespace cbx {
namespace {

constexpr int kOrderThreads = 1024;
constexpr int kBuckets = 256;

// Bucket of cell c, costly cells in the low ones. Any result in range is
// valid (NaN and infinite inputs included): it only orders the work.
__device__ __forceinline__ int cost_bucket(const OrderArgs& a, int c) {
  float lg, per_octave, middle;
  if (a.nops) {
    lg = log2f((float)a.nops[c] + 1.0f);
    per_octave = 16.0f;
    middle = 0.0f;
  } else {
    double av, g0, zeta;
    if (a.track) {
      const double* k0 = a.track + (size_t)c * a.K * 6;
      av = k0[3];
      g0 = k0[4];
      zeta = k0[5];
    } else {
      av = a.phi[c].A_V;
      g0 = a.phi[c].G0;
      zeta = a.phi[c].zeta;
    }
    const double span = (a.t_end_cell ? a.t_end_cell[c] : a.t_end) - a.t0;
    // in logarithms of single precision: exp(-gamma A_V) spans far more than its range
    const float photo = log2f((float)g0) + log2f(a.photo_alpha) - 1.442695f * a.photo_gamma * (float)av;
    const float cosmic = log2f((float)(zeta * 1e17)) + log2f(a.cr_alpha) - 56.4728f;
    const float hi = fmaxf(photo, cosmic), lo = fminf(photo, cosmic);
    lg = hi + log2f(1.0f + exp2f(lo - hi)) + log2f((float)span);
    per_octave = 4.0f;
    middle = 128.0f;
  }
  const float b = (float)(kBuckets - 1) - (lg * per_octave + middle);
  return (int)fminf(fmaxf(b, 0.0f), (float)(kBuckets - 1));  // fmaxf(NaN, 0) = 0
}

__global__ void __launch_bounds__(kOrderThreads) order_cells_kernel(const OrderArgs a) {
  __shared__ int start[kBuckets];
  const int t = threadIdx.x;
  if (t < kBuckets) start[t] = 0;
  __syncthreads();
  for (int c = t; c < a.C; c += kOrderThreads) atomicAdd(&start[cost_bucket(a, c)], 1);
  __syncthreads();
  // exclusive prefix sum over the buckets
  int count = t < kBuckets ? start[t] : 0, sum = count;
  for (int o = 1; o < kBuckets; o <<= 1) {
    const int add = t < kBuckets && t >= o ? start[t - o] : 0;
    __syncthreads();
    sum += add;
    if (t < kBuckets) start[t] = sum;
    __syncthreads();
  }
  if (t < kBuckets) start[t] = sum - count;
  __syncthreads();
  for (int c = t; c < a.C; c += kOrderThreads) a.order[atomicAdd(&start[cost_bucket(a, c)], 1)] = c;
}

}  // namespace

int launch_order(const OrderArgs& a, void* stream) {
  order_cells_kernel<<<1, kOrderThreads, 0, (cudaStream_t)stream>>>(a);
  return cudaGetLastError();
}

}  // namespace cbx
