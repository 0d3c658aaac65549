// The packed layer kernel for 4 pixels per word, 3x3 kernels, one word per kernel row.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

template int launch_strip<4, 3, 1>(const StripLaunch &s, cudaStream_t st);
template int strip_wait_timeouts<4, 3, 1>(unsigned int *h_count);

}  // namespace hikonv
