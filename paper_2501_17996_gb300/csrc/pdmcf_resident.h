// pdmcf_resident.h — resident iteration: many PDHG iterations of one small network in one
// cooperative launch (declarations shared by the driver and the instantiation units).
#pragma once

#include <cuda_runtime.h>

#include "pdmcf_kernels.h"

namespace pdmcf {

// The stop test of Algorithm 2.1 (step 1, evaluated on check iterations), the FP32 rounding
// floor rule (mcf_options.stall_checks) and the rules of the BF16 phase that precedes an FP32
// polish. The driver evaluates them after every chunk, the resident kernel on the device.
struct StopRule {
  int mode = 0;             // MCF_STOP_*
  double eps = 0.0, nm = 0.0;
  int stall_checks = 0;
  double handoff = 0.0;     // > 0: leave once rel_kkt is below it
  int handoff_stall = 0;    // > 0: leave after this many checks without a 5 % improvement
};
struct StopState {
  double floor_best, best_kkt;
  int floor_since, floor_frozen, since_best;
  int verdict;              // StopVerdict
};
enum StopVerdict { STOP_NO = 0, STOP_CONVERGED = 1, STOP_HANDOFF = 2, STOP_STALLED = 3, STOP_NUMERIC = 4 };

inline StopState stop_state_init() {
  StopState s{};
  s.floor_best = s.best_kkt = INFINITY;
  return s;
}

__host__ __device__ inline int stop_test(const DevScalars& h, const StopRule& r, StopState& s) {
  constexpr int kPaper = 0, kKkt = 1;   // MCF_STOP_PAPER, MCF_STOP_REL_KKT
  if (h.numeric_error) return STOP_NUMERIC;
  if (r.mode == kPaper && h.r < r.nm * r.eps) return STOP_CONVERGED;
  if (r.mode == kKkt && h.rel_kkt < r.eps) return STOP_CONVERGED;
  if (r.handoff > 0.0 && h.rel_kkt < r.handoff) return STOP_HANDOFF;
  if (r.mode == kKkt && r.stall_checks > 0 && h.rel_kkt < 100.0 * r.eps) {
    const int frozen = (h.freeze >= 0 && h.freeze <= h.k) ? 1 : 0;
    if (frozen != s.floor_frozen) { s.floor_frozen = frozen; s.floor_best = INFINITY; s.floor_since = 0; }
    if (h.rel_kkt < 0.95 * s.floor_best) { s.floor_best = h.rel_kkt; s.floor_since = 0; }
    else if (++s.floor_since >= r.stall_checks) return STOP_STALLED;
  }
  if (r.handoff_stall > 0) {
    if (h.rel_kkt < 0.95 * s.best_kkt) { s.best_kkt = h.rel_kkt; s.since_best = 0; }
    else if (++s.since_best >= r.handoff_stall) return STOP_HANDOFF;
  }
  return STOP_NO;
}

// Device words of the resident launches; the driver clears `arrived` before each group of
// launches that it queues together.
struct ResidentCtl {
  unsigned arrived;         // grid barrier: CTAs arrived, summed over all barriers of the group
  StopState stop;           // verdict != STOP_NO: the rest of the group returns at once
};

struct ResidentArgs {
  ResidentCtl* ctl;
  long long k;              // first iteration of this launch
  int count;                // iterations of this launch
  int ctas;                 // shares of the work (the grid may be smaller)
  unsigned arrived;         // barrier arrivals of the group's earlier launches
  long long max_iters;      // of the solve; a check falls on multiples of k_check and on the last
  long long k_check;
  StopRule rule;
};

// Variants by row length: a warp owns an edge (`vpt` chunks per lane), a lane `entries` of a piece of
// a node's column; one CTA of 512 threads per SM (128 registers each). Rows longer than eight
// chunks per lane were tried with 384 threads and stay with the per-phase kernels: at n = 3000
// an iteration took 607 us against 367 (twelve warps per SM do not cover the node phase's loads).
struct ResidentVariant { int vpt, entries; };
constexpr int RESIDENT_BLOCK = 512;
constexpr int NUM_RESIDENT = 4;
template <typename P, typename S>
constexpr ResidentVariant resident_variant(int i) {
  constexpr int vpt[NUM_RESIDENT] = {1, 2, 4, 8};
  return {vpt[i], 32 * StoreTraits<S>::VW * vpt[i] <= 512 ? 1 : 2};
}

// `plain` runs iterations without a scalar tail, `special` those with one (a multiple of k_adapt,
// or a stop test).
template <typename P, typename S>
struct ResidentTable {
  void (*plain[NUM_RESIDENT])(IterArgs<P, S>, ResidentArgs);
  void (*special[NUM_RESIDENT])(IterArgs<P, S>, ResidentArgs);
};
const ResidentTable<float, float>& resident_table_f32();
const ResidentTable<double, double>& resident_table_f64();
const ResidentTable<float, __nv_bfloat16>& resident_table_bf16();   // three variants: rows of 1024 entries

// Index of the smallest variant that covers nchunks chunks per row, -1 if none does.
template <typename P, typename S>
inline int pick_resident(int nchunks) {
  for (int t = 0; t < NUM_RESIDENT; ++t)
    if (32 * resident_variant<P, S>(t).vpt >= nchunks) return t;
  return -1;
}

}  // namespace pdmcf
