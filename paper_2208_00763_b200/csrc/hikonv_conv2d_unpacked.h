// Interface between hikonv_conv2d.cu and the one-product-per-multiply comparator (hikonv_conv2d_unpacked.cu).
#pragma once

#include <cuda_runtime.h>

#include "hikonv_internal.h"

namespace hikonv {

struct UnpackedParams {
    const uint32_t *ap;        // codes as int32 [Ci][B*Hp][XBT]
    const uint32_t *wp;        // weights as int32 [Ci*K*K][CoP], kernel rows reversed
    void *out;
    int B, Ci, Co, CoP, K, Ho, Wo, Hp;
    int X;                     // output columns per row
    int XBT;                   // words per row (halo + columns, rounded up so that every tile row can be read in 16-byte pieces)
    int NSEG, XO, XB;          // row segments, output columns per segment (a multiple of 4 when NSEG > 1), positions per segment (XO + K)
    int XBS;                   // words per row in shared memory: 8, 16, 32 or 64
    int TR, TMX, TNX, TCO, CK;
    int a_plane, lead;         // words per channel in shared memory; words before the first row
    int a_words, b_off, b_words;
    int requant, shift, lo, hi;
    int total_rows;            // B * Ho
    int stage_out, WTP, vec, pool, out_signed, out_bits;   // staged output as in the packed layer kernel
    uint32_t mg_xb, mg_ho, mg_xq, mg_ck;
};

struct UnpackedLaunch {
    UnpackedParams p;
    dim3 grid;
    int threads;
    size_t smem_bytes;
};

struct OutputSpec;             // hikonv_conv2d_output.h

// Tiles and parameters of the comparator for a layer; `out` describes the result.
int setup_unpacked(int B, int Ci, int H, int W, int Co, int K, int pad, const OutputSpec &out, const hikonv_tuning_t *tune, int sms,
                   UnpackedLaunch *u);
int launch_unpacked2d(const UnpackedLaunch &u, cudaStream_t st);

}  // namespace hikonv
