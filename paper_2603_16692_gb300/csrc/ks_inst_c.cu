// Kernel instantiations for N = 2^LOGN, LOGN in { 11 }, radix 8, 4 and 16.
#include "ks_rows.cuh"

namespace ks {
#define KS_INST(N, R, C) \
  const LaunchTable &launch_table_##N##_##R##_##C() { return kern::LaunchOne<N, R>::table(); }
KS_INST(11, 3, 0)
KS_INST(11, 2, 0)
KS_INST(11, 4, 0)
#undef KS_INST
}  // namespace ks
