// Two-cells-per-thread step kernels on rows of any length, __nv_bfloat16 storage: the forced collision with unit higher-order rates.
#include "cm_pair.cuh"

namespace cm {
CM_RAGGED_INSTANTIATE_UNIT(__nv_bfloat16)
}  // namespace cm
