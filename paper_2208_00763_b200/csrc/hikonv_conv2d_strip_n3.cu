// The packed layer kernel for words of 3 pixels.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

int launch_strip_n3(const StripLaunch &s, cudaStream_t st) {
    if (s.generic) return launch_strip<3, 0, 0>(s, st);
    if (s.p.K == 3 && s.p.J == 1) return launch_strip<3, 3, 1>(s, st);
    if (s.p.K == 1 && s.p.J == 1) return launch_strip<3, 1, 1>(s, st);
    if (s.p.K == 5 && s.p.J == 2) return launch_strip<3, 5, 2>(s, st);
    return HIKONV_ERR_UNSUPPORTED;
}

}  // namespace hikonv
