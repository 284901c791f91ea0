// Kernel instantiations for N = 2^15.
#include "ks_rows.cuh"

namespace ks {
const LaunchTable &launch_table_15() { return kern::RowFns<15>::table(); }
}  // namespace ks
