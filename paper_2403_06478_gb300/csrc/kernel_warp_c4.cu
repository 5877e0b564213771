// Instantiations of the int32 score kernels and the traceback kernel for 4 band slots per lane (w <= 127).
#include "kernel_lazy32.cuh"
#include "kernel_step.cuh"
#include "kernel_tb.cuh"

namespace agatha {
template cudaError_t launch_warp_c<4, 1>(const DevBatch *, int, cudaStream_t, int, int);
template int occupancy_warp_c<4, 1>();
template cudaError_t launch_step_c<4>(const DevBatch *, int, cudaStream_t, int, int);
template int occupancy_step_c<4>();
template cudaError_t launch_tb_c<4>(const DevBatch *, const TbItem *, int32_t, int32_t *, uint8_t *,
                                    uint32_t *, int32_t *, int, cudaStream_t);
template int occupancy_tb_c<4>();
}  // namespace agatha
