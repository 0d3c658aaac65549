// The packed layer kernel for 2 pixels per word, 3x3 kernels, 2 words per kernel row.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

template int launch_strip<2, 3, 2>(const StripLaunch &s, cudaStream_t st);
template int strip_wait_timeouts<2, 3, 2>(unsigned int *h_count);

}  // namespace hikonv
