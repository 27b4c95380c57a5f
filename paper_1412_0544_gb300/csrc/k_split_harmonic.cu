// k_split_harmonic.cu -- the split FP64 kernels of the harmonic chain (k_split.cuh).
#include "k_split.cuh"

namespace rk4d {
template cudaError_t launch_split_blocked<HARMONIC>(int, int, const BlockedJob &, const CoefD &, cudaStream_t);
template cudaError_t launch_split_persistent<HARMONIC>(int, int, int, const PersistentJob &, const CoefD &, cudaStream_t);
template int persistent_split_max_grid<HARMONIC>(int, int);
}  // namespace rk4d
