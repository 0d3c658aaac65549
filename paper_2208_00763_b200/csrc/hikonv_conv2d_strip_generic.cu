// The packed layer kernel with run-time loop bounds, for every other kernel size and layout.
#include "hikonv_conv2d_strip.cuh"

namespace hikonv {

template int launch_strip<1, 0, 0>(const StripLaunch &s, cudaStream_t st);
template int strip_wait_timeouts<1, 0, 0>(unsigned int *h_count);
template int launch_strip<2, 0, 0>(const StripLaunch &s, cudaStream_t st);
template int launch_strip<3, 0, 0>(const StripLaunch &s, cudaStream_t st);
template int launch_strip<4, 0, 0>(const StripLaunch &s, cudaStream_t st);

// The bounded wait on its own: a barrier that one arrival would complete, and none comes.
__global__ void wait_check_kernel(long long cycles) {
    __shared__ __align__(8) uint64_t barrier;
    const uint32_t bar = smem_address(&barrier);
    mbarrier_init(bar, 1);
    mbarrier_init_fence();
    if (!mbarrier_wait(bar, 0, cycles)) atomicAdd(&strip_timeouts, 1u);
}

int launch_wait_check(long long cycles, cudaStream_t st) { return launch_plain(wait_check_kernel, dim3(1), dim3(1), 0, st, cycles); }

}  // namespace hikonv
