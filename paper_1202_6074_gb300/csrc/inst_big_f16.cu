// Step kernels with 64-bit element offsets (grids with Q * N >= 2^32) for __half storage.
#include "cm_async.cuh"

namespace cm {
template void launch_step_big<__half>(const void*, void*, const void*, const Params&, cudaStream_t);
}  // namespace cm
