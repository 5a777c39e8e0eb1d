// Kernel instantiations: K=9 (557/663/711), radix 2, 8 lanes per frame pair.
#include "vd_variants.cuh"

namespace vd {

template cudaError_t launch_stream_v<9, false, 8>(const StreamParams &, int64_t, bool, cudaStream_t);
template cudaError_t occupancy_wave_v<9, false, 8>(bool, int *);
template cudaError_t launch_batch_v<9, false, 8>(const BatchParams &, int64_t, cudaStream_t);
template cudaError_t occupancy_v<9, false, 8>(int *);
template cudaError_t launch_stream_persistent_v<9, false, 8>(const StreamParams &, int64_t, cudaStream_t);
template cudaError_t occupancy_stream_v<9, false, 8>(int *);

}  // namespace vd
