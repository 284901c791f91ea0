// Kernel instantiations for N = 2^13.
#include "ks_rows.cuh"

namespace ks {
const LaunchTable &launch_table_13() { return kern::RowFns<13>::table(); }
}  // namespace ks
