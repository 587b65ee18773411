// pdmcf_sub.cuh — capped-simplex projection with several rows per warp.
#pragma once

#include "pdmcf_device.cuh"

namespace pdmcf {

// Sums and extrema over the L lanes (a power of two) that own a row; every lane gets them.
template <int L, typename T, typename Op>
__device__ __forceinline__ T lanes_reduce(T v, Op op) {
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// project_mu_n for rows of L < 32 lanes, 32 / L rows per warp: the same iteration, as one loop of
// passes in which each row keeps its own multiplier and state until all rows of the warp are
// done. On short rows a warp per row spends its time in five-step reductions of a few values;
// here a reduction takes log2 L steps and serves 32 / L rows.
template <int L, int N, typename Get>
__device__ __forceinline__ float project_mu_lanes(Get get, float c, float mu0, float lo) {
  auto add = [](float a, float b) { return a + b; };
  auto addi = [](int a, int b) { return a + b; };
  auto mn2 = [](float a, float b) { return fminf(a, b); };
  auto mx2 = [](float a, float b) { return fmaxf(a, b); };
  float mu = mu0 > lo ? mu0 : lo;
  bool done = false, first = true, floor = false;
#pragma unroll 1
  for (int it = 0; it < 67; ++it) {
    float s = 0.f, amin = INFINITY, imax = -INFINITY;
    int n = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float x = get(i);
      if (x > mu) { s += x; ++n; amin = fminf(amin, x); }
      else imax = fmaxf(imax, x);
    }
    s = lanes_reduce<L>(s, add);
    n = lanes_reduce<L>(n, addi);
    amin = lanes_reduce<L>(amin, mn2);
    if (it == 0) imax = lanes_reduce<L>(imax, mx2);
    if (!done) {
      const float phi = s - (float)n * mu - c;
      const float next = n > 0 ? (s - c) / (float)n : lo;   // Newton step
      if (first && phi <= 0.f && mu != lo && phi != 0.f) {  // right of the root
        if (next <= lo) { mu = lo; floor = true; }
        else if (n > 0 && next >= imax) { mu = next; done = true; }   // no inactive entry joins
        else mu = next;
      } else if ((first || floor) && phi <= 0.f) {
        done = true;                                        // at the floor, or at the root
      } else if (n == 0 || !(next > mu)) {
        done = true;
      } else {
        done = next < amin;                                 // no active entry leaves: the root
        mu = next;
        floor = false;
      }
      first = false;
    }
    if (__all_sync(0xffffffffu, done)) break;
  }
  return mu;
}

}  // namespace pdmcf
