// Resident iteration kernels: P = float (iterates), S = __nv_bfloat16 (storage of F).
#include "pdmcf_resident.cuh"

namespace pdmcf {
const ResidentTable<float, __nv_bfloat16>& resident_table_bf16() {
  static const ResidentTable<float, __nv_bfloat16> t = make_resident_table<float, __nv_bfloat16>();
  return t;
}
}  // namespace pdmcf
