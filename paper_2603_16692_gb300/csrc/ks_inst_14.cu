// Kernel instantiations for N = 2^14.
#include "ks_rows.cuh"

namespace ks {
const LaunchTable &launch_table_14() { return kern::RowFns<14>::table(); }
}  // namespace ks
