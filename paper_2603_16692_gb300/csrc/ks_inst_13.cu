// Kernel instantiations for N = 2^13.
#include "ks_fused.cuh"

namespace ks {
const LaunchTable &launch_table_13() { return kern::RowFns<13>::table(); }
const FusedTable &fused_table_13() { return kern::FusedFns<13>::table(); }
}  // namespace ks
