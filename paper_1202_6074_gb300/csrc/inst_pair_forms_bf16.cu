// Two-cells-per-thread step kernels for __nv_bfloat16 storage: the unforced collision with the factorized
// attractor or reduced compressibility fixed at compile time (see cm_pair.cuh).
#include "cm_async.cuh"

namespace cm {
CM_PAIR_INSTANTIATE_FORMS(__nv_bfloat16)
}  // namespace cm
