// Two-cells-per-thread step kernels of the general collision forms for __nv_bfloat16 storage (see cm_pair.cuh).
#include "cm_async.cuh"

namespace cm {
CM_PAIR_INSTANTIATE_GEN(__nv_bfloat16)
}  // namespace cm
