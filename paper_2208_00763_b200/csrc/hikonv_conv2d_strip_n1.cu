// The packed layer kernel for words of 1 pixel.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

int launch_strip_n1(const StripLaunch &s, cudaStream_t st) {
    if (s.generic) return launch_strip<1, 0, 0>(s, st);
    return HIKONV_ERR_UNSUPPORTED;
}

}  // namespace hikonv
