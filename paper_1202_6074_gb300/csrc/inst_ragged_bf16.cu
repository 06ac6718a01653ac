// Two-cells-per-thread step kernels on rows of any length, __nv_bfloat16 storage: the standard collision and the unforced forms.
#include "cm_pair.cuh"

namespace cm {
CM_RAGGED_INSTANTIATE(__nv_bfloat16)
}  // namespace cm
