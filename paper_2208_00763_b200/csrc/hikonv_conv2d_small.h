// Interface between hikonv_conv2d.cu and the one-launch kernel for small layers (hikonv_conv2d_small.cu).
#pragma once

#include "hikonv_conv2d_strip.h"

namespace hikonv {

constexpr int kSmallTM = 2, kSmallTN = 4;      // output rows and channels per thread

struct SmallParams {
    StripParams s;             // geometry, slots and output as for the strip kernel (one row segment; ap, wp and corr unused)
    const int8_t *x, *w;
    int ragged;                // ragged_codes() of x
    int B, H;
    int x_signed, w_signed, Kc;
    int Cz, CF;                // input channels per CTA of a cluster, input channels between two moves
    int ks_log2;               // log2 of the CTAs of a cluster, which share the input channels
    int rows;                  // staged rows of a full CTA
    int col_first;             // image column of slot 0 of the first staged word
    int red_off;               // word offset of the exchange of partial sums
    uint32_t mg_hp, mg_xq, mg_rows;
};

struct SmallLaunch {
    SmallParams p;
    dim3 grid;
    int threads;
    size_t smem_bytes;
    bool sp;
};

int launch_small(const SmallLaunch &l, int N, cudaStream_t st);

}  // namespace hikonv
