// Resident iteration kernels: P = double (iterates), S = double (storage of F).
#include "pdmcf_resident.cuh"

namespace pdmcf {
const ResidentTable<double, double>& resident_table_f64() {
  static const ResidentTable<double, double> t = make_resident_table<double, double>();
  return t;
}
}  // namespace pdmcf
