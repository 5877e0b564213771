// Instantiations of the int32 kernel with 3 warps per pair: 8 and 12 slots per
// lane (frames of 736 and 1,104 slots).
#include "kernel_lazy32.cuh"

namespace agatha {
template cudaError_t launch_warp_c<8, 3>(const DevBatch *, int, cudaStream_t, int, int);
template int occupancy_warp_c<8, 3>();
template cudaError_t launch_warp_c<12, 3>(const DevBatch *, int, cudaStream_t, int, int);
template int occupancy_warp_c<12, 3>();
}  // namespace agatha
