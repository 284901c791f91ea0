// Kernel instantiations for N = 2^14.
#include "ks_fused.cuh"

namespace ks {
const LaunchTable &launch_table_14() { return kern::RowFns<14>::table(); }
const FusedTable &fused_table_14() { return kern::FusedFns<14>::table_inv(); }
}  // namespace ks
