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
// t0) with the network's mean parameters, summed along a track: measured on 150
// species, the mean cost is monotone in it (A_V deciles, 1 Myr: 129, 102, 63 and
// then 26 ms a cell). The reverse sweep's cost is known: the ops on the tape.
// Cells are sorted into 256 logarithmic buckets by one CTA: two passes over the inputs
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

// log2(2^a + 2^b)
__device__ __forceinline__ float log2_sum(float a, float b) {
  const float hi = fmaxf(a, b), lo = fminf(a, b);
  return hi + log2f(1.0f + exp2f(lo - hi));
}

// Photo-reaction and cosmic-ray times per second, as a logarithm of single
// precision: exp(-gamma A_V) spans far more than its range.
__device__ __forceinline__ float log2_rate(const OrderArgs& a, double av, double g0, double zeta) {
  const float photo = log2f((float)g0) + log2f(a.photo_alpha) - 1.442695f * a.photo_gamma * (float)av;
  const float cosmic = log2f((float)(zeta * 1e17)) + log2f(a.cr_alpha) - 56.4728f;
  return log2_sum(photo, cosmic);
}

// The same over a track: up to kTrackKnots of its knots, each for the part of the
// cell's span that it is nearest to. (A cell's first knot alone put those that
// come out of the shade last: 150 species, 760 cells losing 5 mag over 1e5 yr
// took 295 ms, with this 240; gaining them 248 and 254, spread 4.)
constexpr int kTrackKnots = 8;

__device__ float log2_track(const OrderArgs& a, int c, double t_end) {
  const double* knots = a.track + (size_t)c * a.K * 6;
  const int n = min(a.K, kTrackKnots);
  auto knot = [&](int j) { return knots + 6 * (n > 1 ? (size_t)j * (a.K - 1) / (n - 1) : 0); };
  float lg = -INFINITY;
  double from = a.t0;
  for (int j = 0; j < n; ++j) {
    const double* k = knot(j);
    const double to = j + 1 < n ? fmin(fmax(0.5 * (k[0] + knot(j + 1)[0]), from), t_end) : t_end;
    lg = log2_sum(lg, log2_rate(a, k[3], k[4], k[5]) + log2f((float)(to - from)));
    from = to;
  }
  return lg;
}

// Bucket of cell c, costly cells in the low ones. Any result in range is
// valid (NaN and infinite inputs included): it only orders the work.
__device__ __forceinline__ int cost_bucket(const OrderArgs& a, int c) {
  float lg, per_octave, middle;
  if (a.nops) {
    lg = log2f((float)a.nops[c] + 1.0f);
    per_octave = 16.0f;
    middle = 0.0f;
  } else {
    const double t_end = a.t_end_cell ? a.t_end_cell[c] : a.t_end;
    if (a.track)
      lg = log2_track(a, c, t_end);
    else
      lg = log2_rate(a, a.phi[c].A_V, a.phi[c].G0, a.phi[c].zeta) + log2f((float)(t_end - a.t0));
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
