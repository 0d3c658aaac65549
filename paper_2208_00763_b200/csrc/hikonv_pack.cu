// hikonv_pack: Eq. 5, codes -> packed 32- or 64-bit words.
#include "hikonv_cuda.cuh"

namespace hikonv {

// Largest N with a kernel of its own (pack_groups_kernel): the paper's 32-bit configurations hold up to eleven codes.
constexpr int kMaxPackN = 12;

// Four words per thread.  The call is a stream (N bytes in, one word out) and is bound by HBM; with one thread per word
// and byte loads (pack_kernel) it was bound by the N loads per word instead.  Four words take exactly N aligned 32-bit
// words of codes whatever N is, so a thread loads those (16 or 8 bytes at a time where N allows), takes each code out
// with one byte permute, adds it by Horner's rule (one multiply-add per code for 32-bit words) and writes 16-byte
// pieces.  The last, partial group is packed code by code by the thread it falls to.  2^24 4-bit codes, three per 32-bit
// word: 20.5 -> 7.0 us a call among others (39 MB, 5.6 TB/s).
template <bool SIGNED, typename WORD, int N>
__global__ void __launch_bounds__(256) pack_groups_kernel(const int8_t *in, size_t n, int S, WORD *__restrict__ words,
                                                          size_t n_words) {
    grid_dependency_release();
    grid_dependency_wait();
    const size_t g = (size_t)blockIdx.x * 256 + threadIdx.x;
    const size_t x0 = g * 4;
    if (x0 >= n_words) return;
    WORD out[4];
    if ((x0 + 4) * N <= n) {
        uint32_t w[N];
        const int8_t *src = in + x0 * N;
        if constexpr (N % 4 == 0) {
#pragma unroll
            for (int i = 0; i < N; i += 4) {
                const uint4 v = load_ordered(reinterpret_cast<const uint4 *>(src) + i / 4);
                w[i] = v.x; w[i + 1] = v.y; w[i + 2] = v.z; w[i + 3] = v.w;
            }
        } else if constexpr (N % 2 == 0) {
#pragma unroll
            for (int i = 0; i < N; i += 2) {
                const uint2 v = load_ordered(reinterpret_cast<const uint2 *>(src) + i / 2);
                w[i] = v.x; w[i + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) w[i] = load_ordered(reinterpret_cast<const uint32_t *>(src) + i);
        }
        const uint32_t step = sizeof(WORD) == 4 && S < 32 ? 1u << S : 0u;      // S >= 32 only with N == 1
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            WORD a = 0;
#pragma unroll
            for (int i = N - 1; i >= 0; --i) {
                const int e = k * N + i;
                const int32_t v = (int32_t)extract_code<SIGNED>(w[e / 4], e % 4);
                if constexpr (sizeof(WORD) == 4) a = i == N - 1 ? (WORD)v : a * step + (WORD)v;
                else a = i == N - 1 ? (WORD)(long long)v : (a << S) + (WORD)(long long)v;
            }
            out[k] = a;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            WORD a = 0;
            for (int i = 0; i < N; ++i) {
                const size_t idx = (x0 + k) * N + i;
                if (idx < n) a += (WORD)((unsigned long long)(long long)load_code<SIGNED>(in + idx) << (S * i));
            }
            out[k] = a;
        }
    }
    if (x0 + 4 <= n_words) {
        uint4 *dst = reinterpret_cast<uint4 *>(words + x0);
        if constexpr (sizeof(WORD) == 4) {
            *dst = make_uint4((uint32_t)out[0], (uint32_t)out[1], (uint32_t)out[2], (uint32_t)out[3]);
        } else {
            dst[0] = make_uint4((uint32_t)out[0], (uint32_t)((uint64_t)out[0] >> 32), (uint32_t)out[1], (uint32_t)((uint64_t)out[1] >> 32));
            dst[1] = make_uint4((uint32_t)out[2], (uint32_t)((uint64_t)out[2] >> 32), (uint32_t)out[3], (uint32_t)((uint64_t)out[3] >> 32));
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (x0 + k < n_words) words[x0 + k] = out[k];
    }
}

// Any N and any alignment: one thread per word, one byte load per code.
template <bool SIGNED, typename WORD>
__global__ void __launch_bounds__(256) pack_kernel(const int8_t *__restrict__ in, size_t n, int S, int N,
                                                   WORD *__restrict__ words, size_t n_words) {
    const size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n_words) return;
    const size_t base = x * (size_t)N;
    WORD a = 0;
    for (int i = 0; i < N; ++i) {
        const size_t idx = base + i;
        if (idx < n) {
            // two's-complement sum: a negative code borrows from the slots above it, which is
            // what the slot-by-slot decrementer of Eq. 28 builds
            const long long v = code_value<SIGNED>(__ldg(in + idx));
            a += (WORD)((unsigned long long)v << (S * i));
        }
    }
    words[x] = a;
}

template <bool SIGNED, typename WORD, int N = 1>
static int launch_groups(int n_codes, dim3 grid, cudaStream_t st, const int8_t *in, size_t n, int S, WORD *words, size_t n_words) {
    if constexpr (N > kMaxPackN) {
        return HIKONV_ERR_UNSUPPORTED;
    } else {
        if (n_codes == N) return launch_dependent(pack_groups_kernel<SIGNED, WORD, N>, grid, dim3(256), 0, st, in, n, S, words, n_words);
        return launch_groups<SIGNED, WORD, N + 1>(n_codes, grid, st, in, n, S, words, n_words);
    }
}

// The grouped kernel needs the alignment of its widest load and 16-byte aligned output.
template <bool SIGNED, typename WORD>
static int launch_pack(const int8_t *in, size_t n, int S, int N, WORD *words, size_t n_words, cudaStream_t st) {
    const uintptr_t load = N % 4 == 0 ? 16 : N % 2 == 0 ? 8 : 4;
    if (N <= kMaxPackN && (uintptr_t)in % load == 0 && (uintptr_t)words % 16 == 0) {
        const size_t blocks = (n_words + 1023) / 1024;
        if (blocks > 0x7FFFFFFFull) return HIKONV_ERR_UNSUPPORTED;
        return launch_groups<SIGNED, WORD>(N, dim3((unsigned)blocks), st, in, n, S, words, n_words);
    }
    const size_t blocks = (n_words + 255) / 256;
    if (blocks > 0x7FFFFFFFull) return HIKONV_ERR_UNSUPPORTED;
    return launch_plain(pack_kernel<SIGNED, WORD>, dim3((unsigned)blocks), dim3(256), 0, st, in, n, S, N, words, n_words);
}

}  // namespace hikonv

using namespace hikonv;

extern "C" int hikonv_pack(const int8_t *d_in, size_t n, int bits, int is_signed, int S, int N, int word_bits,
                           void *d_words, void *stream) {
    if (!d_in || !d_words) return HIKONV_ERR_INVALID_ARG;
    if (bits < 1 || bits > 8 || S < 1 || N < 1 || (word_bits != 32 && word_bits != 64)) return HIKONV_ERR_INVALID_ARG;
    if (S < bits) return HIKONV_ERR_INVALID_ARG;
    if ((long long)bits + (long long)(N - 1) * S > word_bits) return HIKONV_ERR_NO_FIT;
    if (((uintptr_t)d_words) % (word_bits / 8) != 0) return HIKONV_ERR_INVALID_ARG;
    if (n == 0) return HIKONV_OK;
    const size_t n_words = (n + N - 1) / N;
    cudaStream_t st = (cudaStream_t)stream;
    if (word_bits == 32)
        return is_signed ? launch_pack<true, uint32_t>(d_in, n, S, N, (uint32_t *)d_words, n_words, st)
                         : launch_pack<false, uint32_t>(d_in, n, S, N, (uint32_t *)d_words, n_words, st);
    return is_signed ? launch_pack<true, uint64_t>(d_in, n, S, N, (uint64_t *)d_words, n_words, st)
                     : launch_pack<false, uint64_t>(d_in, n, S, N, (uint64_t *)d_words, n_words, st);
}
