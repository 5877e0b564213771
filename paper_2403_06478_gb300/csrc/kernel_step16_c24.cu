// Instantiations of the 16-bit kernels with a test on every anti-diagonal for
// 24 band slots per lane (w <= 767): score at two register budgets
// (resident blocks per SM), the autotuner's two, and the fused traceback.
#include "kernel_step.cuh"
#include "kernel_tb.cuh"

namespace agatha {
template cudaError_t launch_step16_c<24, 3>(const DevBatch *, int, cudaStream_t, int, int, const int *);
template int occupancy_step16_c<24, 3>();
template cudaError_t launch_step16_c<24, 2>(const DevBatch *, int, cudaStream_t, int, int, const int *);
template int occupancy_step16_c<24, 2>();
template cudaError_t launch_tbs16_c<24, 2>(const DevBatch *, const TbItem *, int32_t, int32_t *, uint8_t *,
                                           uint32_t *, int32_t *, int, cudaStream_t);
template int occupancy_tbs16_c<24, 2>();
}  // namespace agatha
