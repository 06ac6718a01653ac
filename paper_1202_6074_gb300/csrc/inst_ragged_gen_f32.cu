// Two-cells-per-thread step kernels on rows of any length, float storage: the general forms.
#include "cm_pair.cuh"

namespace cm {
CM_RAGGED_INSTANTIATE_GEN(float)
}  // namespace cm
