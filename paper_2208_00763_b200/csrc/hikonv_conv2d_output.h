// What a 2-D layer writes, and how staged rows leave a CTA (shared by the packed kernel and the comparator).
#pragma once

#include <cstdint>

#include "hikonv.h"

namespace hikonv {

struct OutputSpec {
    int requant, shift, lo, hi;
    int pool;                  // 2x2 maximum after requantisation
    int out_bits;              // requantised codes: 8 (one per byte) or 1 / 2 / 4 (dense)
    const void *d_out;         // its alignment decides the width of the stores
    int byte_inputs;           // activations and weights are stored one code per byte, in memory that the outputs do not share: the layer
                               // kernel may read them itself (not what a layer writes, but what decides how it may run)
};

// Output staging of a layer whose row segments hold `seg_cols` output columns: nothing for plain results, which are stored
// directly (staged, plain bytes measured 3 % slower on the 56x56 layer); for dense or pooled codes the bytes per tile row,
// and the widest piece that divides every row start (row width, segment width and the output address).
inline int output_staging(const OutputSpec &o, int Ho, int Wo, int NSEG, int seg_cols, int *stage_out, int *vec) {
    *stage_out = 0;
    *vec = 1;
    if (!o.requant) return (o.pool || o.out_bits != 8) ? HIKONV_ERR_INVALID_ARG : HIKONV_OK;
    if (!o.pool && o.out_bits == 8) return HIKONV_OK;
    if (o.out_bits != 8 && o.out_bits != 4 && o.out_bits != 2 && o.out_bits != 1) return HIKONV_ERR_INVALID_ARG;
    if (o.pool && ((Ho | Wo) & 1)) return HIKONV_ERR_UNSUPPORTED;      // the fused 2x2 pool wants even output sizes
    if (o.out_bits < 8 && (o.lo < (o.lo < 0 ? -(1 << (o.out_bits - 1)) : 0) ||
                           o.hi > (o.lo < 0 ? (1 << (o.out_bits - 1)) - 1 : (1 << o.out_bits) - 1)))
        return HIKONV_ERR_INVALID_ARG;                                  // the clamp range must fit the stored width
    if (o.pool && NSEG > 1 && (seg_cols & 1)) return HIKONV_ERR_UNSUPPORTED;
    *stage_out = 1;
    const int w_out = o.pool ? Wo / 2 : Wo, seg_out = o.pool ? seg_cols / 2 : seg_cols;
    if (o.out_bits == 8) {
        int v = o.pool ? 8 : 16;
        while (v > 1 && (w_out % v != 0 || (NSEG > 1 && seg_out % v != 0) || ((uintptr_t)o.d_out % v) != 0)) v /= 2;
        *vec = v == 2 ? 1 : v;
    } else {
        // rows and row segments must start on byte boundaries of the dense output
        if ((w_out * o.out_bits) % 8 != 0 || (NSEG > 1 && (seg_out * o.out_bits) % 8 != 0)) return HIKONV_ERR_UNSUPPORTED;
        const int row_bytes = w_out * o.out_bits / 8, seg_bytes = seg_out * o.out_bits / 8;
        *vec = (row_bytes % 4 == 0 && (NSEG == 1 || seg_bytes % 4 == 0) && ((uintptr_t)o.d_out % 4) == 0) ? 4 : 1;
    }
    return HIKONV_OK;
}

// Multiple (of 4) that the groups of N columns in a row segment must come in, so that segments of a dense output row start on
// byte boundaries (segment width in codes, halved by the pool, times out_bits a multiple of 8).
inline int segment_multiple(const OutputSpec &o, int N) {
    int mult = 4;
    if (o.requant && o.out_bits < 8 && o.out_bits > 0) {
        const int unit = o.pool ? 16 : 8;
        int g = N * o.out_bits, a = unit;
        while (a) { const int t = g % a; g = a; a = t; }               // g = gcd(N out_bits, unit)
        while (mult % (unit / g) != 0) mult += 4;
    }
    return mult;
}

}  // namespace hikonv
