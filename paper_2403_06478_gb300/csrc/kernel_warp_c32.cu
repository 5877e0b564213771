// Instantiations of the int32 score kernel with a test on every anti-diagonal and of the
// traceback kernel for 32 band slots per lane (w <= 1023).
#include "kernel_step.cuh"
#include "kernel_tb.cuh"

namespace agatha {
template cudaError_t launch_step_c<32>(const DevBatch *, int, cudaStream_t, int, int);
template int occupancy_step_c<32>();
template cudaError_t launch_tb_c<32>(const DevBatch *, const TbItem *, int32_t, int32_t *, uint8_t *,
                                    uint32_t *, int32_t *, int, cudaStream_t);
template int occupancy_tb_c<32>();
}  // namespace agatha
