// pdmcf_flat.h — node phase of iterations without a scalar tail, over (node, column piece) items
// (declarations).
#pragma once

#include "pdmcf_kernels.h"

namespace pdmcf {

constexpr int FLAT_BLOCK = 256;
// Entries per lane of a piece (us per iteration with two and with four: FP32 F, n = 3000, 303 and 310,
// BF16 F, n = 2000, 142 and 129; FP64 is bound by the FP64 unit and takes one).
template <typename P, typename S> constexpr int flat_entries() { return sizeof(P) == 8 ? 1 : sizeof(S) == 2 ? 4 : 2; }
using FlatF32 = void (*)(IterArgs<float, float>);
using FlatBf16 = void (*)(IterArgs<float, __nv_bfloat16>);
using FlatF64 = void (*)(IterArgs<double, double>);
FlatF32 flat_kernel_f32();
FlatBf16 flat_kernel_bf16();
FlatF64 flat_kernel_f64();

}  // namespace pdmcf
