// Instantiations of the 16-bit kernels with a test on every anti-diagonal for
// 16 band slots per lane (w <= 511): score at two register budgets
// (resident blocks per SM), the autotuner's two, and the fused traceback.
#include "kernel_step.cuh"
#include "kernel_tb.cuh"

namespace agatha {
template cudaError_t launch_step16_c<16, 4>(const DevBatch *, int, cudaStream_t, int, int, const int *);
template int occupancy_step16_c<16, 4>();
template cudaError_t launch_step16_c<16, 3>(const DevBatch *, int, cudaStream_t, int, int, const int *);
template int occupancy_step16_c<16, 3>();
template cudaError_t launch_tbs16_c<16, 3>(const DevBatch *, const TbItem *, int32_t, int32_t *, uint8_t *,
                                           uint32_t *, int32_t *, int, cudaStream_t);
template int occupancy_tbs16_c<16, 3>();
}  // namespace agatha
