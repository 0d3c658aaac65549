// Index arithmetic and byte-wise maxima shared by the 2-D kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "hikonv_cuda.cuh"

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

// Byte mask of the bytes of word i (bytes 4 i .. 4 i + 3) whose index lies in [first, last).
__device__ __forceinline__ uint32_t byte_range_mask(int i, int first, int last) {
    const int lo = max(first - 4 * i, 0), n = max(last - 4 * i - lo, 0);
    uint32_t m;
    asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(m) : "r"(8 * lo), "r"(8 * n));      // 8 n bits from bit 8 lo on, clamped to the word
    return m;
}

// For pack_row_words: the number of codes of a tensor at an address that is not a multiple of four or that ends at one, else -1.
__host__ inline int ragged_codes(const void *x, int codes) { return (((uintptr_t)x | (unsigned)codes) & 3) != 0 ? codes : -1; }

// Four packed words (Eq. 5) of N codes each, from column col0 on, of an image row of W one-byte codes: zero outside the row, and
// everywhere when row_in is false (the row is then not read).  The row starts at code `row` of the tensor x.
// off4: a byte repeated four times that is taken from every code inside the columns of the image (in rows that are not read too),
// is_signed: the codes, after that, are signed.
// The codes start at any byte: the N + 1 aligned words around them are loaded (those that hold a code of the row), shifted into
// place, blanked outside the row with one mask per word, and packed by byte permute and Horner's rule.  Where the
// tensor's ends are not aligned, the words that reach outside it are put together from bytes; ragged_codes() says so and is all
// that aligned tensors pay (checked word by word for all of them, the 56x56x64 layer took 85.2 us instead of 84.7).
template <int N>
__device__ __forceinline__ void pack_row_words(const int8_t *x, int row, int ragged, int W, int col0, bool row_in, uint32_t off4, bool is_signed,
                                               int S, uint32_t (&word)[4]) {
    const int off = ((int)(uintptr_t)x + row + col0) & 3;        // of the first code in its aligned word
    const int first = row + col0 - off;                          // code at the start of that word (not in the tensor, where col0 < 0)
    const uint32_t *al = reinterpret_cast<const uint32_t *>(x + first);
    uint32_t v[N + 1];
    if (ragged < 0) {
#pragma unroll
        for (int i = 0; i <= N; ++i) {
            const int c = col0 - off + 4 * i;                    // aligned word i holds the codes of columns c .. c + 3
            v[i] = row_in && c + 3 >= 0 && c < W ? load_ordered(al + i) : 0u;
        }
    } else {
#pragma unroll
        for (int i = 0; i <= N; ++i) {
            const int c = col0 - off + 4 * i;
            v[i] = 0u;
            if (!row_in || c + 3 < 0 || c >= W) continue;
            if (first + 4 * i >= 0 && first + 4 * i <= ragged - 4) v[i] = load_ordered(al + i);
            else
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (c + b >= 0 && c + b < W) v[i] |= (uint32_t)(uint8_t)load_ordered(x + row + c + b) << (8 * b);
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[i] = __funnelshift_r(v[i], v[i + 1], 8 * off);
        if (off4 != 0) v[i] = __vsub4(v[i], off4);
        v[i] &= byte_range_mask(i, -col0, W - col0);
    }
    const uint32_t step = 1u << S, ext = is_signed ? 0x8880u : 0x4440u, rep = is_signed ? 0x1111u : 1u;
    // permute selector of byte b, sign- or zero-extended (see extract_code)
    auto code = [&](int e) { return byte_permute(v[e / 4], 0u, ext + (uint32_t)(e % 4) * rep); };
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t a = code(w * N + N - 1);
#pragma unroll
        for (int n = N - 2; n >= 0; --n) a = a * step + code(w * N + n);
        word[w] = a;
    }
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
