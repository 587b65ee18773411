// Flat node phase, F stored as BF16.
#include "pdmcf_flat.cuh"

namespace pdmcf {
FlatBf16 flat_kernel_bf16() {
  return node_flat_kernel<float, __nv_bfloat16, flat_entries<float, __nv_bfloat16>()>;
}
}  // namespace pdmcf
