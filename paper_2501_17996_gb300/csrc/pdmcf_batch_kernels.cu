// Kernel instantiations of the batched iteration (FP32 iterates).
#include "pdmcf_batch_engine.h"

namespace pdmcf {

template <int IDX>
static void fill_batch(BatchTable& t) {
  constexpr ShapeDesc d = kShapes[IDX];
  constexpr int g = batch_group(IDX);
  constexpr int MB = min_blocks<float, d.vpt, 4, d.block>();
  t.edge[g] = batch_edge_kernel<d.vpt, d.group, d.block, MB>;
  t.block[g] = d.block;
}

const BatchTable& batch_table() {
  static const BatchTable t = [] {
    BatchTable t{};
    t.edge[0] = batch_edge_warp_kernel<false, 256, 3>;
    t.block[0] = 256;
    t.edge[1] = batch_edge_warp_kernel<true, 256, 2>;
    t.block[1] = 256;
    fill_batch<4>(t); fill_batch<5>(t); fill_batch<6>(t); fill_batch<7>(t); fill_batch<8>(t);
    fill_batch<9>(t); fill_batch<10>(t); fill_batch<11>(t); fill_batch<12>(t); fill_batch<13>(t);
    t.node = batch_node_kernel<false>;
    t.node_chk = batch_node_kernel<true>;
    t.check = batch_check_kernel;
    return t;
  }();
  return t;
}

}  // namespace pdmcf
