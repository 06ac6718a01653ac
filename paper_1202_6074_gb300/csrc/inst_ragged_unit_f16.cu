// Two-cells-per-thread step kernels on rows of any length, __half storage: the forced collision with unit higher-order rates.
#include "cm_pair.cuh"

namespace cm {
CM_RAGGED_INSTANTIATE_UNIT(__half)
}  // namespace cm
