// Resident iteration kernels: P = float (iterates), S = float (storage of F).
#include "pdmcf_resident.cuh"

namespace pdmcf {
const ResidentTable<float, float>& resident_table_f32() {
  static const ResidentTable<float, float> t = make_resident_table<float, float>();
  return t;
}
}  // namespace pdmcf
