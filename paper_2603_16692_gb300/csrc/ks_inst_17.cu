// Kernel instantiations for N = 2^17.
#include "ks_rows.cuh"

namespace ks {
const LaunchTable &launch_table_17() { return kern::RowFns<17>::table(); }
}  // namespace ks
