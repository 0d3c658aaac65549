// Index arithmetic and byte-wise maxima shared by the 2-D kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace hikonv {

// n / d for 0 <= n < 2^22 and d > 0 with inv_d = 1.0f / d: the float quotient is off by at most one.
// (The per-thread index arithmetic of a tile would otherwise be some thirty integer divisions.)
__device__ __forceinline__ int small_div(int n, int d, float inv_d) {
    int q = (int)((float)n * inv_d);
    const int r = n - q * d;
    if (r < 0) --q;
    else if (r >= d) ++q;
    return q;
}

// n / d for 0 <= n < 2^16 and 0 < d < 2^16 with magic = ceil(2^32 / d) mod 2^32 (0 stands for d == 1): the high
// word of n * magic is the exact quotient because n (d - 1) < 2^32.
__device__ __forceinline__ int fast_div(int n, uint32_t magic) {
    return magic ? (int)__umulhi((uint32_t)n, magic) : n;
}

// n / d for any 32-bit n and a divisor d >= 1 fixed per launch (division by invariant integers using
// multiplication, Granlund and Montgomery 1994): with L = ceil(log2 d) and m = floor(2^32 (2^L - d) / d) + 1,
// t = mulhi(m, n) and n / d = (t + ((n - t) >> min(L, 1))) >> max(L - 1, 0).  Five instructions instead of the
// twenty-odd of a hardware-less 32-bit division.
struct Div32 {
    uint32_t m, s1, s2;
};
__host__ inline Div32 make_div32(uint32_t d) {
    uint32_t L = 0;
    while (L < 32 && (1ull << L) < d) ++L;
    Div32 r;
    r.m = (uint32_t)(((1ull << 32) * ((1ull << L) - d)) / d + 1);
    r.s1 = L < 1 ? L : 1;
    r.s2 = L > 1 ? L - 1 : 0;
    return r;
}
__device__ __forceinline__ uint32_t div32(uint32_t n, const Div32 &d) {
    const uint32_t t = __umulhi(d.m, n);
    return (t + ((n - t) >> d.s1)) >> d.s2;
}

// Maxima of neighbouring bytes of two rows of eight bytes: four bytes.
template <bool SIGNED>
__device__ __forceinline__ uint32_t pool_pairs(uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1) {
    uint32_t v0 = SIGNED ? __vmaxs4(a0, b0) : __vmaxu4(a0, b0);     // the two rows
    uint32_t v1 = SIGNED ? __vmaxs4(a1, b1) : __vmaxu4(a1, b1);
    v0 = SIGNED ? __vmaxs4(v0, v0 >> 8) : __vmaxu4(v0, v0 >> 8);    // bytes 0 and 2 hold the pair maxima
    v1 = SIGNED ? __vmaxs4(v1, v1 >> 8) : __vmaxu4(v1, v1 >> 8);
    return __byte_perm(v0, v1, 0x6420);
}

}  // namespace hikonv
