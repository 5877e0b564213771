// Instantiation of the 16-bit kernel with a test on every anti-diagonal for 20
// band slots per lane (w <= 638): the pairs of a 24-slot batch whose own band
// fits a 640-slot frame.
#include "kernel_step.cuh"

namespace agatha {
template cudaError_t launch_step16_c<20, 2>(const DevBatch *, int, cudaStream_t, int, int, const int *);
template int occupancy_step16_c<20, 2>();
}  // namespace agatha
