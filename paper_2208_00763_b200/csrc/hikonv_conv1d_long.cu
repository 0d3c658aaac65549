// The 1-D packed kernel for long filters: kernels that are cut into more chunks than the register-resident kernels are built for.
//
// A CTA computes THREADS x R consecutive blocks of N outputs.  It packs the blocks' codes once into shared memory (Eq. 5; four
// words per thread from N aligned 32-bit loads, permutes and multiply-adds), then every thread forms R neighbouring
//     Q_x = bias + sum_j A_{x-j} B_j                                                                   (Eq. 9)
// in registers, four chunks at a time: the R + 3 words they need are read from shared memory (R is odd, so a warp's reads fall
// into different banks) and serve 4 R multiplies.  The part of Q_{x-1} above its N low slots is added to Q_x (Theorem 2) in
// registers, across threads through shared memory; the outputs leave through shared memory in 16-byte pieces.
// What bounds it: instruction issue (4 R wide multiplies and about R + 8 other instructions per four chunks), near the memory
// floor for the shortest filters that come here.  The kernel it replaces for them (one block per lane, a shuffle and a shared
// load per multiply, byte loads) took 18.6 us a call for 4.2 M codes and 31 taps (u4 x s4, N = 3, eleven chunks); this one 6.9.
#include "hikonv_conv1d_run.cuh"

namespace hikonv {

// Threads of a CTA.  At two codes per word half of 256, with twice the CTAs per SM: the same warps, but a barrier holds up four of them and
// the phases of more CTAs (load and pack, multiply, store) lie beside each other.  As graphs, 8 x 8 bits, 24 taps: 300 000 / 1 M / 2 M / 4.2 M
// codes 3.56 / 4.78 / 6.12 / 8.71 -> 3.07 / 4.67 / 5.80 / 7.95 us; 384 signals of 2000 to 4.2 M codes, 9 to 32 taps and eight widths took 0.5 to 16 % less, all of
// them.  At three codes it changed nothing (31 taps 6.93 / 6.93), at four and more it cost 5 % (20 taps at 2 bits 5.15 -> 5.4).
__host__ __device__ constexpr int long_threads(int N) { return N == 2 ? 128 : 256; }
// Resident CTAs that the registers leave room for: a signal of a few million codes is about one wave of them, with a tail of a few per
// cent at five CTAs of 256 threads per SM and none at six, which N = 3 reaches without spilling (4.2 M codes, 12 / 16 / 31 taps:
// 6.3 / 7.0 / 7.7 -> 5.5 / 6.3 / 7.3 us for a launch by itself; the other block sizes lost 2 to 20 % at five or six).
__host__ __device__ constexpr int long_resident(int N) { return N == 3 || N == 2 ? 6 : 3; }
constexpr int kLongJ = (kMaxJ + 3) / 4 * 4;                    // chunks, rounded up to whole groups of four
// Blocks per thread: odd, and at most 28 outputs.
__host__ __device__ constexpr int long_run(int N) { return N == 1 ? 15 : N == 2 ? 11 : N <= 4 ? 7 : N == 5 ? 5 : 3; }

template <int N, bool SP, bool FS>
__global__ void __launch_bounds__(long_threads(N), long_resident(N)) conv1d_long_kernel(const Conv1dTcParams p) {
    constexpr int THREADS = long_threads(N), R = long_run(N), TILE = THREADS * R, FRONT = kLongJ;   // blocks per tile; packed words in front of it
    static_assert(TILE % 4 == 0 && FRONT % 4 == 0 && FRONT > kMaxJ - 1, "groups of four words");
    __shared__ __align__(16) uint32_t s_A[FRONT + TILE];
    __shared__ __align__(16) uint32_t s_B[kLongJ];
    __shared__ uint32_t s_hi[THREADS + 1];                // [1 + t]: what thread t's last block hands on; [0]: the block before the tile
    __shared__ __align__(16) int32_t s_out[TILE * N];
    const int tid = threadIdx.x;
    const long long x0 = (long long)blockIdx.x * TILE;         // first block of the tile
    grid_dependency_release();
    grid_dependency_wait();

    if (tid < kLongJ) {                                        // pack the kernel chunk B_j (Eq. 5 on g); zero past the last
        uint32_t b = 0;
        for (int k = 0; k < p.Kc; ++k) {
            const int idx = tid * p.Kc + k;
            if (idx < p.K) {
                const int8_t raw = load_ordered(p.g + idx);
                b += (uint32_t)(p.g_signed ? (int32_t)raw : (int32_t)(uint8_t)raw) << (p.S * k);
            }
        }
        s_B[tid] = b;
    }
    const uint32_t step = 1u << p.S;
    for (int q = tid; q < (FRONT + TILE) / 4; q += THREADS) {
        const long long e0 = (x0 - FRONT + 4 * q) * N;         // first code of the four words
        uint32_t w[N];
        if (p.aligned && e0 >= 0 && e0 + 4 * N <= p.len) {
            const uint32_t *src = reinterpret_cast<const uint32_t *>(p.f + e0);
#pragma unroll
            for (int i = 0; i < N; ++i) w[i] = load_ordered(src + i);
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                uint32_t v = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const long long e = e0 + 4 * i + b;
                    if (e >= 0 && e < p.len) v |= (uint32_t)(uint8_t)load_ordered(p.f + e) << (8 * b);   // Eq. 2: zero outside
                }
                w[i] = v;
            }
        }
        uint32_t a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            a[k] = extract_code<FS>(w[(k * N + N - 1) / 4], (k * N + N - 1) % 4);
#pragma unroll
            for (int n = N - 2; n >= 0; --n) a[k] = a[k] * step + extract_code<FS>(w[(k * N + n) / 4], (k * N + n) % 4);
        }
        *reinterpret_cast<uint4 *>(s_A + 4 * q) = make_uint4(a[0], a[1], a[2], a[3]);
    }
    __syncthreads();

    const uint64_t bias = SP ? p.bias : 0ull;                  // unsigned products are never negative: every slot bias is zero
    uint64_t acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = bias;
    const uint32_t *a_own = s_A + FRONT + tid * R;
    for (int j0 = 0; j0 < p.J; j0 += 4) {
        const uint4 b4 = *reinterpret_cast<const uint4 *>(s_B + j0);
        const uint32_t b[4] = {b4.x, b4.y, b4.z, b4.w};
        uint32_t a[R + 3];                                     // a[i] = A of block (own first) + i - 3 - j0
#pragma unroll
        for (int i = 0; i < R + 3; ++i) a[i] = a_own[i - 3 - j0];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < R; ++r) mad_wide<SP>(acc[r], a[r + 3 - j], b[j]);
    }
    s_hi[1 + tid] = shr64_lo(acc[R - 1], p.hi_shift);
    if (tid == 0) {                                            // the block in front of the tile
        uint64_t q = bias;
        for (int j = 0; j < p.J; ++j) mad_wide<SP>(q, s_A[FRONT - 1 - j], s_B[j]);
        s_hi[0] = shr64_lo(q, p.hi_shift);
    }
    __syncthreads();
    uint32_t carry = s_hi[tid];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint64_t d = acc[r] + carry;
        carry = shr64_lo(acc[r], p.hi_shift);
#pragma unroll
        for (int m = 0; m < N; ++m) {
            const int32_t field = (int32_t)(shr64_lo(d, p.S * m) & p.mask);
            s_out[(tid * R + r) * N + m] = SP ? field - p.carry_bias[m] : field;
        }
    }
    __syncthreads();
    const long long y0 = x0 * N;
    if (p.aligned && y0 + TILE * N <= p.n_out) {
        int4 *dst = reinterpret_cast<int4 *>(p.y + y0);
        for (int i = tid; i < TILE * N / 4; i += THREADS) __stcs(dst + i, reinterpret_cast<const int4 *>(s_out)[i]);
    } else {
        for (int i = tid; i < TILE * N; i += THREADS)
            if (y0 + i < p.n_out) p.y[y0 + i] = s_out[i];
    }
}

template <int N>
static int launch_long_n(const Conv1dTcParams &p, bool sp, bool fs, cudaStream_t st) {
    const long long per_tile = (long long)long_threads(N) * long_run(N) * N;
    const long long tiles = (p.n_out + per_tile - 1) / per_tile;
    if (tiles > 0x7FFFFFFFLL) return HIKONV_ERR_UNSUPPORTED;
    const dim3 grid((unsigned)tiles), block(long_threads(N));
    if (!sp) return launch_dependent(conv1d_long_kernel<N, false, false>, grid, block, 0, st, p);
    if (fs) return launch_dependent(conv1d_long_kernel<N, true, true>, grid, block, 0, st, p);
    return launch_dependent(conv1d_long_kernel<N, true, false>, grid, block, 0, st, p);
}

bool conv1d_long_available(int N) { return N >= 1 && N <= 8; }

int launch_conv1d_long(const Conv1dTcParams &p, int N, bool sp, bool fs, cudaStream_t st) {
    switch (N) {
        case 1: return launch_long_n<1>(p, sp, fs, st);
        case 2: return launch_long_n<2>(p, sp, fs, st);
        case 3: return launch_long_n<3>(p, sp, fs, st);
        case 4: return launch_long_n<4>(p, sp, fs, st);
        case 5: return launch_long_n<5>(p, sp, fs, st);
        case 6: return launch_long_n<6>(p, sp, fs, st);
        case 7: return launch_long_n<7>(p, sp, fs, st);
        case 8: return launch_long_n<8>(p, sp, fs, st);
        default: return HIKONV_ERR_UNSUPPORTED;
    }
}

}  // namespace hikonv
