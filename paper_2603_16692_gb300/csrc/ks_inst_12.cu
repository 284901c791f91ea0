// Kernel instantiations for N = 2^12.
#include "ks_fused.cuh"

namespace ks {
const LaunchTable &launch_table_12() { return kern::RowFns<12>::table(); }
const FusedTable &fused_table_12() { return kern::FusedFns<12>::table(); }
}  // namespace ks
