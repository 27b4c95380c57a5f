// k_split_roessler.cu -- the split FP64 kernels of the roessler chain (k_split.cuh).
#include "k_split.cuh"

namespace rk4d {
template cudaError_t launch_split_blocked<ROESSLER>(int, int, const BlockedJob &, const CoefD &, cudaStream_t);
template cudaError_t launch_split_persistent<ROESSLER>(int, int, int, const PersistentJob &, const CoefD &, cudaStream_t);
template int persistent_split_max_grid<ROESSLER>(int, int);
}  // namespace rk4d
