// Interface between hikonv_conv2d.cu and the kernel that packs the weights of several filters (hikonv_conv2d_filters.cu).
#pragma once

#include <cuda_runtime.h>

#include "hikonv_internal.h"

namespace hikonv {

constexpr int kFiltersThreads = 256;     // most threads of a CTA
constexpr int kFiltersK = 3;             // kernel size
constexpr int kFiltersSlots = 3;         // filters in a word
constexpr int kFiltersSlotBits = 17;     // bits of a slot: three of them in the 52 bits of a double's fraction

struct FiltersParams {
    const int8_t *x, *w;
    void *out;
    int codes;                           // of x, all of them
    int B, Ci, H, W, Co, pad, Ho, Wo;
    int Hp;                              // padded rows per image
    int SH, strips;                      // pairs of output rows per image, in the layer
    int tiles, NSEG, TQ, TS;             // tiles of the layer (a CTA takes every gridDim.x-th), row segments, pairs of output columns per segment, row pairs per CTA
    int pos_warps, groups;               // warps per set of positions, groups of words
    int WT;                              // words per CTA
    int CK, rows, PW, plane;             // input channels per step, staged rows, codes per staged row, codes per channel
    uint32_t mg_tq, mg_sh, mg_hp;   // fast_div() multipliers
    int x_signed, w_signed;
    int slot_bias;                       // of a slot: what lifts its most negative sum to 0
    double bias;                         // the biases of all slots of a word
    int requant, shift, lo, hi, pool, pair_stores;
};

struct FiltersLaunch {
    FiltersParams p;
    dim3 grid;
    int threads;
    size_t smem_bytes;
    int NW;                              // words per thread: 2, 4 or 6
};

// CTAs of kFiltersThreads that fit an SM by their registers.
__host__ __device__ constexpr int filters_resident(int NW) { return NW >= 4 ? 2 : 3; }

int launch_filters(const FiltersLaunch &l, cudaStream_t st);

}  // namespace hikonv
