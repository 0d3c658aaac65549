// The packed layer kernel for words of 2 pixels.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

int launch_strip_n2(const StripLaunch &s, cudaStream_t st) {
    if (s.generic) return launch_strip<2, 0, 0>(s, st);
    if (s.p.K == 3 && s.p.J == 2) return launch_strip<2, 3, 2>(s, st);
    if (s.p.K == 3 && s.p.J == 1) return launch_strip<2, 3, 1>(s, st);
    if (s.p.K == 1 && s.p.J == 1) return launch_strip<2, 1, 1>(s, st);
    if (s.p.K == 5 && s.p.J == 3) return launch_strip<2, 5, 3>(s, st);
    return HIKONV_ERR_UNSUPPORTED;
}

}  // namespace hikonv
