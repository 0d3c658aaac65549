// Interface between hikonv_conv2d.cu (planning, packing launch, entry points) and the packed layer kernel
// (hikonv_conv2d_strip.cuh, instantiated per layout by hikonv_conv2d_strip_*.cu: pixels per word, kernel size, words per row).
#pragma once

#include <cuda_runtime.h>

#include "hikonv_internal.h"

namespace hikonv {

constexpr int kStripThreads = 256;   // most threads of a CTA
constexpr int kStripBPitch = 32;     // words per packed kernel row in shared memory (TCO or more)
constexpr int kStripMaxCK = 16;      // most input channels of a stage and thread group
constexpr int kStripMaxGroups = 4;   // most thread groups that share the input channels of a tile

struct StripParams {
    const uint32_t *ap;              // packed activations [Ci][B * Hp][XBT]
    const uint32_t *wp;              // packed weights [Ci * K * J][CoP]
    void *out;
    int Ci, Co, CoP, K, J, Ho, Wo;
    int Hp, ap_rows, XBT;            // packed rows per image, rows per channel (B * Hp), words per row
    int SH, strips;                  // strips (TM output rows) per image, strips of the layer
    int NSEG, XO, XB, halo;          // row segments, output groups per segment, positions per segment and strip, 1: position 0 only feeds its neighbour
    int X, col_off;                  // output groups per row; slot m of group x is output column x N + m - col_off
    int pitch;                       // words per staged activation row (XB + J - 1 rounded up to a multiple of 4)
    int TS, TNX, TCO, CK;            // strips and channel lanes per CTA, channels per CTA, input channels per stage
    int run, runs_per_move;          // input channels between two possible moves (CK or less), such runs between two moves
    int plane;                       // words between two channels of a staged activation tile
    int a_words, b_off, b_words;     // words per staged activation tile, offset of the first weight tile, words per weight tile
    int bar_off, e_off;              // word offsets of the two mbarriers and of the second accumulators
    uint32_t mg_xb, mg_sh;           // fast_div() multipliers: XB, SH
    // slots: S bits each; every slot starts at bias and moves its bits above the low h to a second accumulator
    int S, SN, h;                    // slot width, S N, h
    uint64_t bias, mask_low, mask_high;
    uint32_t slot_mask;
    int32_t slot_bias[8];            // bias of slot m (0 beyond the last)
    int up_slots;                    // slots above the N low ones
    // output
    int requant, shift, lo, hi;
    int stage_out, pool, out_bits, out_signed, vec, WTP, tile_off;   // pool: 0, 1, or 2 where the stored bytes do not keep the order of the codes
    const int32_t *corr;             // x_off * (sum of a channel's weights over the taps 0 .. k), [K][CoP]; null when x_off == 0
    int W, pad;
};

struct StripLaunch {
    StripParams p;
    dim3 grid;
    int threads;
    size_t smem_bytes;
    int TM, TN, KS;                  // output rows and channels per thread, thread groups that share the input channels
    bool sp;                         // signed product
    bool moves;                      // the layer needs the second accumulator
    bool generic;                    // the kernel with run-time loop bounds
};

// Thread tiles the kernel is built for: 4 x 8, 2 x 8 and 2 x 4 rows x channels.  4 x 4 was as fast as 2 x 8 on no layer.
inline bool strip_tile_built(int TM, int TN) { return (TM == 2 && (TN == 4 || TN == 8)) || (TM == 4 && TN == 8); }
// Tiles that are also built with two or four thread groups, which share the input channels.
inline bool strip_split_built(int TM, int TN, int KS, bool generic) { return !generic && TM == 2 && (KS == 2 || (KS == 4 && TN == 4)); }
// 8-byte entries of a thread in the second-accumulator area: TM TN and one that keeps the pitch odd.
__host__ __device__ constexpr int strip_e_pitch(int TM, int TN) { return TM * TN + 1; }
// Is there a kernel with unrolled loops for (N, K, J), and does it add the upper slots to the next word while packed?
inline bool strip_unrolled(int N, int K, int J) {
    if (K == 1) return J == 1 && N >= 2 && N <= 4;
    if (K == 3) return (J == 1 && N >= 2 && N <= 4) || (J == 2 && N == 2);
    if (K == 5) return (N == 4 && J <= 2) || (N == 3 && J == 2) || (N == 2 && J == 3);
    return false;
}
constexpr bool strip_packed_add(int N, int K, int J) {
    return K > 0 && !(J == 1 && K == N + 1) && !(N == 4 && K == 5);
}

// Explicitly instantiated, one layout per file: (N, 0, 0) with run-time bounds, (N, K, J) for strip_unrolled ones.
template <int N, int KT, int JT>
int launch_strip(const StripLaunch &s, cudaStream_t st);
// Threads of the layout's kernels on the current device whose bounded wait for a stage of operands ran out (the generic kernels
// share the counter of N = 1).  Reads a device variable: the caller synchronises.
template <int N, int KT, int JT>
int strip_wait_timeouts(unsigned int *h_count);
// Launches one thread that waits `cycles` for a barrier of its own which nothing completes and counts that wait with the generic kernels'.
int launch_wait_check(long long cycles, cudaStream_t st);

}  // namespace hikonv
