// Two-cells-per-thread step kernels on rows of any length, __nv_bfloat16 storage: the general forms.
#include "cm_pair.cuh"

namespace cm {
CM_RAGGED_INSTANTIATE_GEN(__nv_bfloat16)
}  // namespace cm
