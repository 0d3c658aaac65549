// The packed layer kernel with run-time loop bounds, for every other kernel size and layout.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

template int launch_strip<1, 0, 0>(const StripLaunch &s, cudaStream_t st);
template int strip_wait_timeouts<1, 0, 0>(unsigned int *h_count);
template int launch_strip<2, 0, 0>(const StripLaunch &s, cudaStream_t st);
template int launch_strip<3, 0, 0>(const StripLaunch &s, cudaStream_t st);
template int launch_strip<4, 0, 0>(const StripLaunch &s, cudaStream_t st);

}  // namespace hikonv
