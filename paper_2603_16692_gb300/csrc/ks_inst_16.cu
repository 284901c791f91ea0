// Kernel instantiations for N = 2^16.
#include "ks_rows.cuh"

namespace ks {
const LaunchTable &launch_table_16() { return kern::RowFns<16>::table(); }
}  // namespace ks
