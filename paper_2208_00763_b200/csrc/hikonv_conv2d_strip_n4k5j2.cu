// The packed layer kernel for 4 pixels per word, 5x5 kernels, 2 words per kernel row.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

template int launch_strip<4, 5, 2>(const StripLaunch &s, cudaStream_t st);
template int strip_wait_timeouts<4, 5, 2>(unsigned int *h_count);

}  // namespace hikonv
