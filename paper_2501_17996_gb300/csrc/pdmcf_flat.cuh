// pdmcf_flat.cuh — node phase of one iteration (Zhang & Boyd, Algorithm 2.1, step 2) over (node,
// column piece) items.
#pragma once

#include "pdmcf_flat.h"
#include "pdmcf_resident.cuh"

namespace pdmcf {

// Node phase of an iteration without a scalar tail: the resident iteration's pieces (node_pieces),
// column block by column block. A row of F is gathered by its head and by its tail; within a block
// both reads fall into the same few megabytes of F, so the second hits L2 where a pass node by
// node read it from HBM again, and a thread has one chunk of a column instead of all of them.
// n = 3000, m = 24 000 (FP32, log): 130 us, with DRAM and issue slots at 44 % each, two FP32
// entries per lane (node_kernel without in-sums: 138 us); n = 1000 FP64 with an exponent per
// pair: 2.5 -> 1.2 ms per iteration, bound by the FP64 unit.
template <typename P, typename S, int N>
__global__ void __launch_bounds__(FLAT_BLOCK, sizeof(P) == 8 ? 2 : 3)
node_flat_kernel(const __grid_constant__ IterArgs<P, S> a) {
  constexpr int NW = FLAT_BLOCK / 32;
  const unsigned warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, nwarps = gridDim.x * NW;
  const unsigned pieces = (unsigned)a.n * ((unsigned)(a.ld + 32 * N - 1) / (32 * N));
  if (warp >= pieces) return;
  NodePiece q;
  NodeItem<P, N> x;
  node_place<P, S, N>(a, warp, q);
  q.edge = node_edge(a, q, (int)(threadIdx.x & 31));
  node_data<P, S, N>(a, q, x);
  node_state<P, S, N>(a, a.parity, q, x);
  double acc[NODE_PARTS] = {0.0};
  node_pieces<P, S, N, false>(a, a.parity, warp, pieces, nwarps, q, x, (P)a.sc->beta, acc);
  // a sum that is not finite is reported as the scalar tail would
  if (!isfinite(acc[0])) a.sc->numeric_error = 1;
}

}  // namespace pdmcf
