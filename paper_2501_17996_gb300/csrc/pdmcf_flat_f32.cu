// Flat node phase, F stored as FP32, and in FP64.
#include "pdmcf_flat.cuh"

namespace pdmcf {
FlatF32 flat_kernel_f32() { return node_flat_kernel<float, float, flat_entries<float, float>()>; }
FlatF64 flat_kernel_f64() { return node_flat_kernel<double, double, flat_entries<double, double>()>; }
}  // namespace pdmcf
