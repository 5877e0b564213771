// Instantiations of the int32 score kernel with a test on every anti-diagonal and of the
// traceback kernel for 24 band slots per lane (w <= 767).
#include "kernel_step.cuh"
#include "kernel_tb.cuh"

namespace agatha {
template cudaError_t launch_step_c<24>(const DevBatch *, int, cudaStream_t, int, int);
template int occupancy_step_c<24>();
template cudaError_t launch_tb_c<24>(const DevBatch *, const TbItem *, int32_t, int32_t *, uint8_t *,
                                    uint32_t *, int32_t *, int, cudaStream_t);
template int occupancy_tb_c<24>();
}  // namespace agatha
