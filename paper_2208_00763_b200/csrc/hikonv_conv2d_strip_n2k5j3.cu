// The packed layer kernel for 2 pixels per word, 5x5 kernels, 3 words per kernel row.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

template int launch_strip<2, 5, 3>(const StripLaunch &s, cudaStream_t st);
template int strip_wait_timeouts<2, 5, 3>(unsigned int *h_count);

}  // namespace hikonv
