// Two-cells-per-thread step kernels on rows of any length, __half storage: the standard collision and the unforced forms.
#include "cm_pair.cuh"

namespace cm {
CM_RAGGED_INSTANTIATE(__half)
}  // namespace cm
