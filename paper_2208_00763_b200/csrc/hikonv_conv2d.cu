// hikonv_conv2d: a convolution layer as row-wise packed 1-D convolutions (Theorem 3).  This file plans a layer, packs its
// operands and holds the entry points; the layer kernel is in hikonv_conv2d_strip.cuh, the one-product-per-multiply comparator
// in hikonv_conv2d_unpacked.cu.
//
// Activations are packed once per layer by pack_operands_kernel into Ap[ci][b*Hp + hp][xb] (zero padding rows and columns
// materialised), weights by the same launch into Bw[(ci,kh,j)][co].  Layers with unsigned activations and signed weights may be
// packed as x - 2^(p-1), the padding rows included, and get 2^(p-1) times the sum of the weights that meet a column of the image
// back in the epilogue (plan_layer says when and why).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "hikonv_cuda.cuh"
#include "hikonv_conv2d_filters.h"
#include "hikonv_conv2d_output.h"
#include "hikonv_conv2d_small.h"
#include "hikonv_conv2d_strip.h"
#include "hikonv_conv2d_unpacked.h"
#include "hikonv_conv2d_util.cuh"

namespace hikonv {

// Reversed, packed kernel rows (Theorem 3: g = W[co][ci][kh][K-1:0], then Eq. 5 per chunk of Kc taps).
// wp[((ci*K + kh)*J + j)*CoP + co] = sum_{k' < Kc} g[j Kc + k'] 2^(S k').  For the comparator S == 0,
// Kc == 1: one int32 weight per word.
struct WeightPackParams {
    const int8_t *w;
    uint32_t *wp;
    int Co, Ci, K, J, Kc, S, w_signed, CoP;
    int w_bits;                // storage: 8 = one code per byte, 1 / 2 / 4 = dense (8 / w_bits codes per byte)
    int w_blocks;              // CTAs that pack kernel rows, one word per thread; the CTAs before them sum the weights of a channel each (x_off != 0)
    Div32 d_cg, d_j;           // divisions by the number of groups of eight channels and by J
    int x_off;                 // offset taken from every activation code (0: none)
    int32_t *corr;             // corr[k][co] = x_off * sum of channel co's weights over ci, kh and kw <= k; K rows of CoP entries
};

// Code number e of a tensor stored densely with `bits` (1, 2, 4 or 8) bits per code: code e occupies bits
// [(e bits) % 8, (e bits) % 8 + bits) of byte (e bits) / 8, two's complement when signed (Section V-B: weights and
// features kept compressed in memory and unpacked as they are read).
__device__ __forceinline__ int32_t load_dense_code(const int8_t *base, size_t e, int bits, bool is_signed) {
    const size_t bit = e * (size_t)bits;
    const uint32_t byte = (uint8_t)load_ordered(base + (bit >> 3));
    const uint32_t v = (byte >> (int)(bit & 7)) & ((1u << bits) - 1u);
    const uint32_t sb = 1u << (bits - 1);
    return is_signed ? (int32_t)((v ^ sb) - sb) : (int32_t)v;
}

// A warp packs four neighbouring (row, chunk) words of eight channels: a channel's rows are contiguous in memory and the
// words are contiguous over channels, so a load touches eight sectors and a store four.  (With 32 channels per warp every
// lane's loads touched a sector of its own; with the sums below taken one load at a time, the packing launch of the
// 256 -> 256 channel layer on 64 14x14 maps took 15.2 us, now 9.8.)
__device__ __forceinline__ void pack_weight_words(const WeightPackParams &q, int warp, int lane) {
    const int rg = (int)div32((uint32_t)warp, q.d_cg), cg = warp - rg * ((q.CoP + 7) / 8);
    const int rj = rg * 4 + (lane >> 3), co = cg * 8 + (lane & 7);
    if (rj >= q.Ci * q.K * q.J || co >= q.CoP) return;
    const int row = (int)div32((uint32_t)rj, q.d_j), j = rj - row * q.J;
    uint32_t word = 0;
    if (co < q.Co) {
        const size_t row_e = ((size_t)co * q.Ci * q.K + row) * q.K;              // first code of the kernel row
        for (int k = 0; k < q.Kc; ++k) {
            const int g_idx = j * q.Kc + k;                                      // index into the reversed row
            if (g_idx < q.K) {
                int32_t v;
                if (q.w_bits == 8) {
                    const int8_t raw = load_ordered(q.w + row_e + (q.K - 1 - g_idx));
                    v = q.w_signed ? (int32_t)raw : (int32_t)(uint8_t)raw;
                } else {
                    v = load_dense_code(q.w, row_e + (q.K - 1 - g_idx), q.w_bits, q.w_signed != 0);
                }
                word += (uint32_t)v << (q.S * k);
            }
        }
    }
    q.wp[(size_t)rj * q.CoP + co] = word;
}

// corr[k][co] = x_off * sum_{ci, kh, kw <= k} W[co][ci][kh][kw], k < K: one CTA per output channel, so that the few loads
// of a thread are all in flight together (one warp per channel, a load at a time, was the longest part of the launch).
template <int CTAS>
__device__ __forceinline__ void sum_channel_weights(const WeightPackParams &q, int co, int tid) {
    __shared__ int32_t s_part[8][4];
    const int rows = q.Ci * q.K;
    int32_t run = 0;                                                 // thread 0: the sum over the taps done
    for (int k0 = 0; k0 < q.K; k0 += 4) {
        int32_t sum[4] = {0, 0, 0, 0};
        if (co < q.Co) {
#pragma unroll(CTAS == 3 ? 4 : 1)
            for (int r = tid; r < rows; r += 256) {
                const size_t e = ((size_t)co * rows + r) * q.K + k0;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k0 + k < q.K) {
                        if (q.w_bits == 8) {
                            const int8_t raw = load_ordered(q.w + e + k);
                            sum[k] += q.w_signed ? (int32_t)raw : (int32_t)(uint8_t)raw;
                        } else {
                            sum[k] += load_dense_code(q.w, e + k, q.w_bits, q.w_signed != 0);
                        }
                    }
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sum[k] = __reduce_add_sync(0xFFFFFFFFu, sum[k]);
            if ((tid & 31) == 0) s_part[tid >> 5][k] = sum[k];
        }
        __syncthreads();
        if (tid == 0) {
            for (int k = 0; k < 4 && k0 + k < q.K; ++k) {
                for (int w = 0; w < 8; ++w) run += s_part[w][k];
                q.corr[(size_t)(k0 + k) * q.CoP + co] = run * q.x_off;
            }
        }
        __syncthreads();
    }
}

// Packed activation rows (Eq. 5): ap[(ci * B*Hp + b*Hp + hp) * XBT + xb] packs the N input pixels of padded row hp that
// start at column col_first + xb N (input row hp - pad), zero where the row or a column lies outside the image.  For the
// comparator S == 0 and N == 1: one int32 code per word.
// One thread packs four consecutive words of a row (one 16-byte store); threads are numbered through all
// (ci, b) planes, so that small maps still fill their CTAs.  The first CTAs of the launch sum the channels' weights
// (when the layer runs on shifted codes) and pack the kernel rows, so that a layer needs one
// packing launch and its longest serial work starts first.
// The 4 N codes of a thread start at any byte: it loads the N + 1 aligned words around them, shifts them into place, blanks
// the bytes outside the row with one mask per word and packs by byte permute and Horner's rule (as hikonv_pack does).
// x_bits: storage of the activations, 8 = one code per byte, 1 / 2 / 4 = dense (code by code).
// With wq.x_off != 0 the slots of the image's columns hold code - x_off, in the padding rows too (code 0 there); slots left and
// right of the image hold 0.  XS: the packed values are signed.
struct ActPackDivs {
    Div32 per_plane, b, xq;    // pieces per (ci, b) plane, images, 16-byte pieces per packed row
};

// CTAS: CTAs that fit an SM by their registers.  The loads of a thread come in one group and all of a CTA's together, so a large
// launch wants as many warps as an SM holds: with three CTAs (80 registers) the first layer of the compact CNN (4984 CTAs) took
// 17.2 us, with eight 10.7 (32 images of 64x56x56: 11.4 and 7.6).  A launch of few CTAs starts while the kernel before it still
// runs, and with eight they pile up on the SMs that are free first: 24x45x61 and 48x37x53 layers took 31.1 and 27.2 us a call
// instead of 29.8 and 26.3.
template <bool XS, int N, int CTAS>
__global__ void __launch_bounds__(256, CTAS) pack_operands_kernel(const int8_t *x, int ragged, int B, int Ci, int H,
                                                            int W, int Hp, int pad, int col_first, int S, int XBT,
                                                            uint32_t *__restrict__ ap, int weight_blocks, const WeightPackParams wq,
                                                            int x_bits, const ActPackDivs dv, unsigned act_items) {
    grid_dependency_release();
    grid_dependency_wait();                                          // the input may come from the kernel before; the workspace may still be read by it
    // the first CTAs sum the channels' weights (the longest serial work of the launch) and pack the kernel rows
    if ((int)blockIdx.x < weight_blocks) {
        const int cb = weight_blocks - wq.w_blocks;                  // CTAs that sum weights (0 unless x_off != 0)
        if ((int)blockIdx.x < cb) sum_channel_weights<CTAS>(wq, (int)blockIdx.x, (int)threadIdx.x);
        else pack_weight_words(wq, ((int)blockIdx.x - cb) * 8 + ((int)threadIdx.x >> 5), (int)threadIdx.x & 31);
        return;
    }
    // the (plane, piece) pairs are numbered through: a CTA may span several small planes (ci * B + b)
    const int xq = XBT / 4;                                          // 16-byte pieces per packed row
    const int per_plane = Hp * xq;
    const unsigned item = (blockIdx.x - (unsigned)weight_blocks) * 256u + threadIdx.x;
    if (item >= act_items) return;
    const int plane = (int)div32(item, dv.per_plane);
    const int piece = (int)(item - (unsigned)plane * (unsigned)per_plane);
    const int ci = (int)div32((uint32_t)plane, dv.b), b = plane - ci * B;
    const int hp = (int)div32((uint32_t)piece, dv.xq), q = piece - hp * xq;
    const int hi = hp - pad;
    uint32_t word[4] = {0u, 0u, 0u, 0u};
    const int col0 = col_first + 4 * q * N;                          // input column of slot 0 of the first word
    const bool row_in = hi >= 0 && hi < H;
    if ((row_in || wq.x_off != 0) && col0 + 4 * N > 0 && col0 < W) {
        const int row_e = ((b * Ci + ci) * H + (row_in ? hi : 0)) * W;   // first code of the input row (below 2^31)
        if (x_bits == 8) {
            pack_row_words<N>(x, row_e, ragged, W, col0, row_in, (uint32_t)wq.x_off * 0x01010101u, XS, S, word);
        } else {
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    const int col = col0 + w * N + n;
                    if (col >= 0 && col < W) {
                        const int32_t code = row_in ? load_dense_code(x, (size_t)(row_e + col), x_bits, XS && wq.x_off == 0) : 0;
                        word[w] += (uint32_t)(code - wq.x_off) << (S * n);
                    }
                }
        }
    }
    *reinterpret_cast<uint4 *>(ap + ((size_t)plane * Hp + hp) * XBT + 4 * q) = make_uint4(word[0], word[1], word[2], word[3]);
}

// VEC input bytes of two rows per thread (VEC = 8: two 8-byte loads, one 4-byte store; VEC = 16: two
// 16-byte loads, one 8-byte store), per-byte maxima; needs W % VEC == 0 and VEC-byte aligned input,
// VEC/2-byte aligned output.
template <bool SIGNED, int VEC>
__global__ void __launch_bounds__(256) maxpool2x2_vec_kernel(const int8_t *in, long long items, int H, int W,
                                                             int8_t *__restrict__ out) {
    grid_dependency_release();
    grid_dependency_wait();
    const int Ho = H / 2, WV = W / VEC;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < items; idx += (long long)gridDim.x * blockDim.x) {
        const int wv = (int)(idx % WV);
        const long long rest = idx / WV;
        const int ho = (int)(rest % Ho);
        const long long c = rest / Ho;
        const int8_t *src = in + (c * H + 2 * ho) * (long long)W + VEC * wv;
        int8_t *dst = out + (c * Ho + ho) * (long long)(W / 2) + (VEC / 2) * wv;
        if constexpr (VEC == 16) {
            const uint4 r0 = load_ordered(reinterpret_cast<const uint4 *>(src));
            const uint4 r1 = load_ordered(reinterpret_cast<const uint4 *>(src + W));
            *reinterpret_cast<uint2 *>(dst) = make_uint2(pool_pairs<SIGNED>(r0.x, r0.y, r1.x, r1.y), pool_pairs<SIGNED>(r0.z, r0.w, r1.z, r1.w));
        } else {
            const uint2 r0 = load_ordered(reinterpret_cast<const uint2 *>(src));
            const uint2 r1 = load_ordered(reinterpret_cast<const uint2 *>(src + W));
            *reinterpret_cast<uint32_t *>(dst) = pool_pairs<SIGNED>(r0.x, r0.y, r1.x, r1.y);
        }
    }
}

__global__ void __launch_bounds__(256) maxpool2x2_kernel(const int8_t *__restrict__ in, int BC, int H, int W, int is_signed,
                                                         int8_t *__restrict__ out) {
    const int Ho = H / 2, Wo = W / 2;
    const long long total = (long long)BC * Ho * Wo;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long long)gridDim.x * blockDim.x) {
        const int wo = (int)(idx % Wo);
        const long long rest = idx / Wo;
        const int ho = (int)(rest % Ho);
        const long long c = rest / Ho;
        const int8_t *src = in + (c * H + 2 * ho) * W + 2 * wo;
        int v[4] = {src[0], src[1], src[W], src[W + 1]};
        if (!is_signed) {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] &= 0xFF;
        }
        out[idx] = (int8_t)max(max(v[0], v[1]), max(v[2], v[3]));
    }
}

// ------------------------------------------------------------------ host side

struct Conv2dSetup {
    hikonv_layout_t L;
    bool unpacked;
    bool one_launch;      // the kernel for small layers, which packs its operands itself
    SmallLaunch small;
    bool filters;         // the kernel whose words hold the weights of several filters
    FiltersLaunch filt;
    StripLaunch strip;    // the packed kernel, or
    UnpackedLaunch un;    // the comparator
    // packed operands in the workspace: weights [Ci K J][CoP], x_off corrections [K][CoP], activations [Ci][B Hp][XBT]
    int CoP, Hp, XBT, col_first, x_off;
    size_t corr_off, wp_bytes, ap_words;
    double positions;     // words multiplied per (ci, kh, j) and output channel, in two launches
    int small_blocks;     // words per row in the one-launch kernel
};

static int sm_count() {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

constexpr int kSmemPerSm = 228 * 1024;   // shared memory of an SM; every resident CTA takes 1 KB more than it asks for
constexpr int kSmemPerCta = 227 * 1024;

// A layer as the tile choice sees it.
struct StripProblem {
    int B, Ci, Co, Ho, Wo, N, K, J, pad;
    int CF, max_moves;          // input channels between two moves, moves the second accumulator takes
    int split_moves[kStripMaxGroups + 1];   // most moves that so many groups sharing the input channels may make together (0: their sums may not be added)
    bool moves, generic;
    bool requant, pool;
    int xo_mult;
    int sms;
};

struct StripChoice {
    int TM, TN, TNX, KS, TS, NSEG, XO, XB, halo, X, col_off, pitch, CK, run, runs_per_move, plane, bar_off, e_off, threads;
    size_t smem;
    long long ctas;
    double cost;
};

// Staged rows of TS strips.
static int staged_rows(int TS, int TM, int SH, int Hp, int K) {
    const int gap = Hp - SH * TM;                                    // rows between the strips of one image and the next, beyond TM per strip
    const int crossings = (TS - 1 + SH - 1) / SH;
    return TS * TM + K - 1 + std::max(0, crossings * gap);
}

// Completes a candidate (TM, TN, TNX, TS and the row cut are set) and models its time in scheduler cycles of the busiest SM:
// issue cycles of a warp (4.3 per multiply, about one for every other instruction; a tile of 2 x 4 costs a tenth more per multiply
// than 4 x 8 by this count and by the clock) times the warps of the busiest scheduler, wave by wave.  Returns false when the candidate cannot run.
// most_resident: the CTAs of an SM that share its memory, at most.
static bool complete_choice(const StripProblem &q, StripChoice *c, int most_resident = 32) {
    const int SH = ceil_div(q.Ho, c->TM), Hp = q.Ho + q.K - 1, KJ = q.K * q.J;
    const long long strips = (long long)q.B * SH;
    c->pitch = (c->XB + q.J - 1 + 3) / 4 * 4;
    const int rows = staged_rows(c->TS, c->TM, SH, Hp, q.K);
    c->plane = rows * c->pitch;
    c->threads = (c->TS * c->XB * c->TNX + 31) / 32 * 32 * c->KS;
    if (c->threads > kStripThreads) return false;
    const int warps = c->threads / 32, TCO = c->TNX * c->TN;
    c->ctas = (strips + c->TS - 1) / c->TS * c->NSEG * ceil_div(q.Co, TCO);
    const int share = (int)std::min<long long>(1000000, (c->ctas + q.sms - 1) / q.sms);
    // channels per stage: as many as leave room for the CTAs that the registers allow; runs of CF channels that fill stages
    const int by_regs = std::min(65536 / (c->threads * 128), most_resident);
    const int want = std::max(1, std::min(by_regs, share));
    const size_t e_bytes = q.moves ? (size_t)c->threads * strip_e_pitch(c->TM, c->TN) * 8 : 0;
    const size_t per_cta = std::min<size_t>(kSmemPerCta, kSmemPerSm / want - 1024);
    if (per_cta < e_bytes + 4096) return false;
    const size_t room = per_cta - e_bytes - 64;
    // CK: channels of a stage and group
    const int Cg = ceil_div(q.Ci, c->KS);
    int CK = (int)std::min<size_t>(std::min(std::min(kStripMaxCK, 32 / c->KS), Cg), room / (2 * 4 * (size_t)c->KS * (c->plane + KJ * kStripBPitch)));
    if (CK < 1) return false;
    c->run = CK;
    c->runs_per_move = 1;
    if (q.moves) {
        if (q.CF <= CK) {
            c->run = q.CF;
            CK = CK / q.CF * q.CF;
        } else {
            // several stages per move, as close to CF channels as stages of nearly CK fill it (the second accumulator has room for
            // ceil(Ci / CF) moves and a little more)
            int best = 0, best_ck = 1;
            for (int ck = CK; ck >= 1; --ck) {
                const int eff = q.CF / ck * ck;
                if (eff > best && (best == 0 || 2 * ck > CK || ceil_div(q.Ci, best) > q.max_moves)) { best = eff; best_ck = ck; }
            }
            CK = best_ck;
            c->runs_per_move = q.CF / CK;
            c->run = CK;
        }
        // each of several groups also makes a move after its last channel, and their second accumulators are added
        if (c->KS > 1 && c->KS * ceil_div(Cg, c->run * c->runs_per_move) > q.split_moves[c->KS]) return false;
    }
    const double warp_ci = Cg;                                       // input channels that a warp goes through
    CK *= c->KS;
    c->CK = CK;
    size_t words = 2 * (size_t)CK * (c->plane + KJ * kStripBPitch);
    const size_t xch = (size_t)warps * c->TNX * c->TM * c->TN / c->KS * 2, sums = c->KS > 1 ? (size_t)c->threads * c->TM * c->TN * 2 : 0;
    const int rps = q.pool ? c->TM / 2 : c->TM;
    const size_t tile = (xch + 3) / 4 * 4 + (size_t)TCO * c->TS * rps * ((c->XO * q.N + 15) / 16 * 16) / 4;
    words = (std::max(words, std::max(xch + sums, tile)) + 3) / 4 * 4;
    c->bar_off = (int)words;
    c->e_off = (int)words + 4;
    c->smem = words * 4 + 16 + e_bytes;
    if (c->smem > (size_t)kSmemPerCta) return false;
    const int resident = std::max(1, std::min(by_regs, (int)(kSmemPerSm / (c->smem + 1024))));
    // issue cycles of one warp
    const double mt = (double)c->TM * c->TN;
    double per_ch = 4.3 * mt * KJ + 0.5 * (c->TM + q.K - 1) * q.J + 0.6 * KJ * c->TN / 4 + 8 + 80.0 * c->KS / CK;
    if (q.generic) per_ch += KJ * 16.0;
    if (q.moves) per_ch += 10.0 * mt / q.CF;
    const double split = q.moves ? 6.0 * q.N + 12 : 3.0 * q.N + 6;
    double fixed = 400 + mt / c->KS * (split + q.N * (q.pool ? 4.0 : q.requant ? 6.0 : 3.0));
    if (c->KS > 1) fixed += 100 + mt * (q.moves ? 18.0 : 6.0);
    const double warp_cycles = warp_ci * per_ch + fixed;
    // n resident CTAs of this size on an SM
    // (few warps hide less of each other's latencies: two per scheduler took a sixth longer than eight, by the clock over 17 layers)
    auto cycles_of = [&](double n) {
        const double per_scheduler = n * ceil_div(warps, 4);
        return std::max(per_scheduler, 1.5) * (1.0 + 0.3 / per_scheduler) * warp_cycles + 1500 + 250.0 * q.Ci / CK;
    };
    const double slots = (double)resident * q.sms, waves = c->ctas / slots;
    double cycles;
    if (waves <= 1.0) cycles = cycles_of(share);
    else if (waves < 3.0) {
        const double full = std::floor(waves);
        const double rest = std::ceil((c->ctas - full * slots) / q.sms);
        cycles = full * cycles_of(resident) + (rest > 0 ? cycles_of(rest) : 0.0);
    } else cycles = (waves + 0.35) * cycles_of(resident);
    // With run-time bounds the tile of 2 x 8 is the fastest oftener than this count says, in small CTAs above all (by the clock over 24
    // layers of 2x2 to 9x9 kernels the choice is 1.8 % off the best tile, 3 % without these two).
    if (q.generic) cycles *= (c->TM == 4 ? 1.1 : 1.0) * (waves > 1.0 ? 1.0 + 0.1 * (1.0 / resident - 0.5) : 1.0);
    // Where CTAs follow one another, more and smaller ones on an SM cover each other's barriers: at costs within half a per cent, four
    // CTAs of 128 threads took 5 to 6 % less than two of 256 (32x64x56x56 -> 64 at 8 bits unsigned 241.6 -> 229.6 us, signed 228.0 ->
    // 220.5; 16x24x56x61 -> 256 6 x 4 bits 141.6 -> 126.4).  Enough to decide between tiles of equal cost: with more of it the 4-bit
    // 56x56 layer took 91 us instead of 84.
    if (waves > 1.0 && !q.generic) cycles *= 1.0 + 0.03 * (1.0 / resident - 0.5);
    c->cost = cycles;
    return true;
}

// Chooses the thread tile, thread groups, channel lanes, row cut and strips per CTA.  force_*: 0 = free.
static StripChoice choose_strips(const StripProblem &q, int force_tm, int force_tn, int force_ks, int force_tnx, int force_rows) {
    static const int tiles[6][3] = {{4, 8, 1}, {2, 8, 1}, {2, 4, 1}, {2, 8, 2}, {2, 4, 2}, {2, 4, 4}};
    StripChoice best;
    std::memset(&best, 0, sizeof(best));
    best.cost = -1.0;
    const int c0 = q.K - 1 - q.pad;
    if (q.generic && force_tm == 4) force_tn = 0;                 // (taken as before with any number of channels)
    for (const auto &tile : tiles) {
        const int TM = tile[0], TN = tile[1], KS = tile[2];
        if (KS > 1 && (!strip_split_built(TM, TN, KS, q.generic) || q.Ci < 2 * KS || (q.moves && q.split_moves[KS] == 0))) continue;
        if (force_ks > 0 && KS != force_ks && !q.generic) continue;
        if (!strip_tile_built(TM, TN) || (force_tm > 0 && TM != force_tm) || (force_tn > 0 && TN != force_tn)) continue;
        if (TN == 8 && q.Co <= 4 && force_tn != 8 && force_tm != 4) continue;      // (four rows are built with eight channels only)
        const int SH = ceil_div(q.Ho, TM);
        const long long strips = (long long)q.B * SH;
        for (int TNX = 1; TNX * TN <= kStripBPitch; TNX *= 2) {
            if (force_tnx > 0 ? TNX != std::min(force_tnx, kStripBPitch / TN) : (TNX > 1 && TNX * TN / 2 >= q.Co)) continue;
            const int maxpos = kStripThreads / (TNX * KS);
            // uncut rows start at the image's first column (a word then holds no padding but the row's end); the positions of a
            // cut row need the word in front of them, and its segments start at columns XO N
            int tried = 0;
            for (int cut = 1; cut <= 4096 && tried < 3; ++cut) {
                StripChoice c;
                c.TM = TM; c.TN = TN; c.TNX = TNX; c.KS = KS;
                if (cut == 1) {
                    c.NSEG = 1; c.halo = 0; c.col_off = c0;
                    c.X = c.XO = c.XB = ceil_div(q.Wo + c0, q.N);
                } else {
                    c.halo = 1; c.col_off = 0;
                    c.X = ceil_div(q.Wo, q.N);
                    c.XO = (ceil_div(c.X, cut) + q.xo_mult - 1) / q.xo_mult * q.xo_mult;
                    c.NSEG = ceil_div(c.X, c.XO);
                    c.XB = c.XO + 1;
                    if (c.NSEG < 2) break;
                }
                if (c.XB > maxpos) {
                    cut = std::max(cut, c.XB / maxpos - 1);          // on to the cuts that may fit
                    continue;
                }
                if (cut > 1 && c.XO < 24 && best.cost >= 0) break;     // narrow segments only where nothing else fits
                ++tried;
                const int ts_hi = (int)std::max<long long>(1, std::min<long long>(maxpos / c.XB, strips));
                // a forced height stands for itself, or for the greatest below it that fits
                const bool forced = force_rows > 0;
                for (int TS = forced ? std::min(ceil_div(force_rows, TM), ts_hi) : 1; TS >= 1 && TS <= ts_hi; TS += forced ? -1 : 1) {
                    c.TS = TS;
                    bool fits = complete_choice(q, &c);
                    for (int resident = 16; forced && !fits && resident >= 1; resident /= 2) fits = complete_choice(q, &c, resident);
                    if (!fits) continue;
                    if (best.cost < 0 || c.cost < best.cost * (1.0 - 1e-9)) best = c;
                    if (forced) break;
                }
            }
        }
    }
    return best;
}

// The one-launch kernel for small layers: its tile and cut of the input channels, and the modelled cycles of the call.
struct SmallChoice {
    int TNX, TS, ks_log2, Cz, rows, XB, pitch, threads;
    size_t words;
    long long ctas;
    double cost;
};

static SmallChoice choose_small(const StripProblem &q) {
    SmallChoice best;
    std::memset(&best, 0, sizeof(best));
    best.cost = -1.0;
    constexpr int TM = kSmallTM, TN = kSmallTN;
    const int SH = ceil_div(q.Ho, TM), Hp = q.Ho + q.K - 1, KJ = q.K * q.J;
    const long long strips = (long long)q.B * SH;
    SmallChoice c;
    c.XB = ceil_div(q.Wo + q.K - 1 - q.pad, q.N);
    c.pitch = (c.XB + q.J - 1 + 3) / 4 * 4;
    // not worth looking at beyond a few million multiplies per SM
    if ((double)strips * c.XB * q.Co * q.Ci * KJ * TM > 3.0e6 * q.sms) return best;
    for (c.TNX = 1; c.TNX <= 8; c.TNX *= 2) {
        const int TCO = c.TNX * TN;
        if (c.TNX > 1 && TCO / 2 >= q.Co) break;
        for (c.TS = 1; c.TS * c.XB * c.TNX <= kStripThreads && c.TS <= strips; ++c.TS) {
            c.threads = (c.TS * c.XB * c.TNX + 31) / 32 * 32;
            c.rows = staged_rows(c.TS, TM, SH, Hp, q.K);
            const int warps = c.threads / 32, per_sched = ceil_div(warps, 4);
            const long long tiles = (strips + c.TS - 1) / c.TS * ceil_div(q.Co, TCO);
            for (c.ks_log2 = 0; c.ks_log2 <= (q.pool ? 2 : 3); ++c.ks_log2) {
                const int ks = 1 << c.ks_log2;
                if (ks > q.Ci) break;
                c.Cz = ceil_div(q.Ci, ks);
                c.ctas = tiles * ks;
                const double a_items = (double)c.Cz * c.rows * (c.pitch / 4), b_items = (double)c.Cz * KJ * TCO;
                if (a_items >= 65536.0) continue;
                const size_t stage = (size_t)c.Cz * ((size_t)c.rows * c.pitch + KJ * kStripBPitch);
                const size_t xch = (size_t)warps * c.TNX * TM * TN * 2, red = ks > 1 ? (size_t)c.threads * TM * TN * q.N : 0;
                const size_t tile = q.pool ? (size_t)TCO * c.TS * ((c.XB * q.N + 15) / 16 * 16) / 4 : 0;
                c.words = (std::max(stage, xch + red + tile) + 3) / 4 * 4;
                if (c.words * 4 > (size_t)(kSmemPerCta - 1024)) continue;
                const int resident = std::max(1, std::min(std::min(65536 / (c.threads * 128), (int)(kSmemPerSm / (c.words * 4 + 1024))), 32));
                const long long share = (c.ctas + q.sms - 1) / q.sms;
                const double waves = std::ceil((double)share / resident), at_once = (double)std::min<long long>(share, resident) * per_sched;
                const double mul = 4.3 * TM * TN * KJ;
                const double pack = (std::ceil(a_items / c.threads) * 75 + std::ceil(b_items / c.threads) * (25 + 8 * q.K)) * at_once + 1800;
                const double mults = c.Cz * std::max(at_once * (mul + 30 + (q.moves ? 80.0 / q.CF : 0)), mul + 120 + (q.moves ? 200.0 / q.CF : 0));
                const double split = at_once * TM * TN * 14 * q.N + 500 + (ks > 1 ? 2000 + 60.0 * ks : 0);
                c.cost = 4000 + waves * (pack + mults + split);
                if (best.cost < 0 || c.cost < best.cost) best = c;
            }
        }
    }
    return best;
}

constexpr int kFiltersMaxCi = 6, kFiltersMinCo = 16;    // see plan_layer
constexpr double kFiltersMinOutputs = 1.0e6;

// The kernel whose words hold the weights of several filters: its tile and the modelled SM cycles of the call.  The model is a sum: the launch,
// the packing of the kernel words, the first fetch, then per tile the double-precision pipe (2.1 cycles a multiply-add; 190 per word for
// the split; 119 per channel and row of four codes staged), a third of the passes through shared memory, and per channel and
// step what a CTA waits for (latencies, the barrier).  Fitted to 3531 tiles of 237 layers (1 to 6 input channels, 16 to 128
// filters, 1 to 1024 images, 4 to 1080 rows): 6 % rms.  The tiles it picks are 1.4 % slower than the best measured ones on average; a maximum of
// pipe and latency in place of the sum picked tiles 5.7 % slower, and left some layers up to 29 % slower than in two launches.
struct FiltersChoice {
    int NW, groups, TQ, NSEG, TS, pos_warps, CK, rows, PW, threads;
    size_t smem;
    long long tiles, gx, gy;
    double cost;
};

// What tune->tile forces of it: words per thread, groups of words, input channels per step, most CTAs that share the tiles (0: free).
struct FiltersForced {
    int NW, groups, CK, ctas;
};

static FiltersChoice choose_filters(const StripProblem &q, const FiltersForced &force) {
    FiltersChoice best;
    std::memset(&best, 0, sizeof(best));
    best.cost = -1.0;
    constexpr int K = kFiltersK, KK = K * K, NS = kFiltersSlots;
    const int SH = ceil_div(q.Ho, 2), QT = ceil_div(q.Wo, 2), Hp = q.Ho + K - 1;
    FiltersChoice c;
    const long long strips = (long long)q.B * SH;
    const int words = ceil_div(q.Co, NS);
    static const int word_tiles[3] = {6, 4, 2};
    for (int NW : word_tiles)
        for (c.groups = 1; c.groups <= 8 && (c.groups == 1 || (c.groups - 1) * NW < words); c.groups *= 2) {
            if ((force.NW > 0 && NW != force.NW) || (force.groups > 0 && c.groups != force.groups)) continue;
            c.NW = NW;
            const int warps_max = kFiltersThreads / 32 / c.groups, WT = NW * c.groups;
            const size_t word_bytes = 8 * (size_t)q.Ci * KK * WT;
            c.gy = ceil_div(words, WT);
            int last_tq = 0;
            for (int cut = 1; cut <= ceil_div(QT, 32); ++cut) {
                // whole rows, or segments of whole warps of pixel pairs
                c.NSEG = cut;
                c.TQ = ceil_div(QT, cut);
                if (cut > 1) {
                    c.TQ = (c.TQ + 31) / 32 * 32;
                    c.NSEG = ceil_div(QT, c.TQ);
                }
                if (c.TQ == last_tq) continue;
                last_tq = c.TQ;
                if (c.TQ > warps_max * 32) continue;
                // a warp's multiply-adds and split
                const double products = q.Ci * KK * 4.0 * NW * 2.1 + 190.0 * NW;
                auto hopeless = [&](double cycles) { return best.cost >= 0 && 2530 + cycles * (1.0 - 1e-9) >= best.cost; };
                if (hopeless((double)(strips * c.NSEG * c.TQ * c.groups * c.gy) / (128.0 * q.sms) * products)) continue;
                const int ts_hi = (int)std::max<long long>(1, std::min<long long>(warps_max * 32 / c.TQ, strips));
                for (c.TS = 1; c.TS <= ts_hi; ++c.TS) {
                    c.pos_warps = ceil_div(c.TS * c.TQ, 32);
                    c.threads = c.pos_warps * 32 * c.groups;
                    c.rows = staged_rows(c.TS, 2, SH, Hp, K);
                    c.PW = (2 * c.TQ + K - 1 + 3) / 4 * 4;
                    c.tiles = (strips + c.TS - 1) / c.TS * c.NSEG;
                    const int by_regs = std::min(filters_resident(NW) * (kFiltersThreads / c.threads), 8);
                    const size_t plane = 8 * (size_t)c.rows * c.PW;
                    const double items = (double)c.rows * (c.PW / 4) / c.threads;      // rows of four codes that a thread stages per channel
                    const int per_sched = ceil_div(c.threads / 32, 4);
                    // of a tile, by itself, and for every CTA that shares the SM
                    const double busy = per_sched * (products + 119.0 * q.Ci * items) + 0.36 * (c.threads / 32) * q.Ci * (32 + KK * NW / 2.0 + 8 * items);
                    auto waits = [&](int CK) { return 294.0 * q.Ci + 1020.0 * ceil_div(q.Ci, CK); };
                    // what comes before the first tile, with n warps on a scheduler: packing the kernel words, fetching the first step's CK channels
                    const double word_rounds = std::ceil((double)q.Ci * KK * WT / (4.0 * c.threads));
                    auto before = [&](double n, int CK) { return word_rounds * (1520 + 175 * n) + std::ceil(CK * items / 2.0) * 440; };
                    if (hopeless(before(per_sched, 1) + (double)(c.tiles * c.gy) / q.sms * busy + waits(q.Ci))) continue;
                    for (int want = 1; want <= by_regs; ++want) {
                        if (want > 1 && c.tiles * c.gy <= (long long)(want - 1) * q.sms) break;
                        c.gx = std::max<long long>(1, std::min<long long>(c.tiles, (long long)want * q.sms / c.gy));
                        if (force.ctas > 0) c.gx = std::min<long long>(c.gx, force.ctas);
                        const long long per_cta = (c.tiles + c.gx - 1) / c.gx;
                        c.gx = (c.tiles + per_cta - 1) / per_cta;
                        const double resident = std::max(1.0, std::min((double)want, std::ceil((double)(c.gx * c.gy) / q.sms)));
                        const double rounds = std::ceil((double)(c.gx * c.gy) / (resident * q.sms));
                        const double n = resident * per_sched, tiles_of_sm = rounds * per_cta;
                        if (hopeless(before(n, 1) + tiles_of_sm * (resident * busy + waits(q.Ci)))) continue;
                        const size_t room = std::min<size_t>(kSmemPerCta, kSmemPerSm / want - 1024);
                        for (int part = 1, CK = 0; part <= 8; part *= 2) {
                            const int divided = force.CK > 0 ? std::min(force.CK, q.Ci) : ceil_div(q.Ci, part);
                            if (CK == divided) continue;
                            CK = divided;
                            const size_t smem = word_bytes + 2 * CK * plane;
                            if (smem > room) continue;
                            c.cost = 2530 + before(n, CK) + tiles_of_sm * (resident * busy + waits(CK));
                            c.CK = CK;
                            c.smem = smem;
                            if (best.cost < 0 || c.cost < best.cost * (1.0 - 1e-9)) best = c;
                        }
                    }
                }
            }
        }
    return best;
}

static int plan_layer(int B, int Ci, int H, int W, int Co, int K, int stride, int pad, int p, int q, int xs, int ws,
                      const OutputSpec &out, int algo, const hikonv_tuning_t *tune, Conv2dSetup *s) {
    if (B < 1 || Ci < 1 || H < 1 || W < 1 || Co < 1 || K < 1 || K > kMaxK) return HIKONV_ERR_INVALID_ARG;
    if (validate_codes(p, q) != HIKONV_OK) return HIKONV_ERR_INVALID_ARG;
    if (stride != 1 || pad < 0 || pad >= K) return HIKONV_ERR_UNSUPPORTED;
    if (algo == HIKONV_ALGO_PACKED64EMU || algo == HIKONV_ALGO_DP4A) return HIKONV_ERR_UNSUPPORTED;
    if (algo != HIKONV_ALGO_PACKED32 && algo != HIKONV_ALGO_UNPACKED_IMAD) return HIKONV_ERR_INVALID_ARG;
    if (out.requant && (out.shift < 0 || out.shift > 31 || out.lo < -128 || out.hi > 255 || out.lo > out.hi)) return HIKONV_ERR_INVALID_ARG;
    const int Ho = H + 2 * pad - K + 1, Wo = W + 2 * pad - K + 1;
    if (Ho < 1 || Wo < 1) return HIKONV_ERR_INVALID_ARG;
    if (Ho >= 60000) return HIKONV_ERR_UNSUPPORTED;              // the kernels divide row numbers below 2^16 by a multiply (fast_div)
    if ((double)B * Ci * H * W >= 2147483647.0 || (double)B * Ho >= 2147483647.0) return HIKONV_ERR_UNSUPPORTED;
    // the exact sums must fit int32
    const double max_code = (double)(1 << p) * (double)(1 << q);
    if ((double)Ci * K * K * max_code >= 1073741824.0) return HIKONV_ERR_UNSUPPORTED;

    s->unpacked = (algo == HIKONV_ALGO_UNPACKED_IMAD);
    const int own_xs = xs;                                       // (layers on shifted codes change xs)
    s->CoP = (Co + 3) / 4 * 4;
    s->Hp = Ho + K - 1;
    s->x_off = 0;
    s->one_launch = false;
    s->filters = false;
    hikonv_layout_t &L = s->L;
    if (s->unpacked) {
        std::memset(&L, 0, sizeof(L));
        L.N = 1; L.S = 0; L.Kc = 1; L.J = K; L.segments = 1; L.top_bits = 32; L.M = Ci * K; L.signed_prod = (xs || ws) ? 1 : 0;
        const int rc = setup_unpacked(B, Ci, H, W, Co, K, pad, out, tune, sm_count(), &s->un);
        if (rc != HIKONV_OK) return rc;
        s->XBT = s->un.p.XBT;
        s->col_first = K - 1 - pad - K;
        s->positions = (double)s->un.p.total_rows * s->un.p.NSEG * s->un.p.XB;
    } else {
        int rc = make_layout(p, q, xs, ws, K, 2, Ci * K, Wo, tune, &L);
        if (rc != HIKONV_OK) return rc;
        // Unsigned activations against signed weights: the products of codes x - 2^(p-1) span about half the range,
        // so a slot takes nearly twice as many of them between two carry-save moves, or a word one more pixel (5-bit
        // codes: three instead of two).  Layers whose signed layout is cheaper by the estimate below run on the shifted codes and get
        // 2^(p-1) * (sum of the channel's weights) added back in the epilogue: from 128 input channels on always, from 32 on
        // when the layer is large enough to fill the device.
        const double threads4_own = (double)B * Ho * (ceil_div(Wo, L.N) + L.J) / 4 * ceil_div(Co, 4);
        const bool small_layer = threads4_own <= 1.1 * sm_count() * 2 * kStripThreads;
        if (!xs && ws) {
            hikonv_layout_t Ls;
            // issue cycles per pixel and (ci, kh) pair: J multiplies of about four cycles and, every M pairs, a move of
            // about thirteen, shared by the N pixels of a word; the shifted codes are taken for a gain of 7 % or more,
            // always when they put more pixels into a word, else under the depth conditions above
            auto cycles = [&](const hikonv_layout_t &l) { return (l.J * 4.1 + 13.0 / std::min(l.M, Ci * K)) / l.N; };
            // (not with one tap per word, which only a forced layout has: the corrections would not fit the workspace)
            if (make_layout(p, q, 1, ws, K, 2, Ci * K, Wo, tune, &Ls) == HIKONV_OK && (K == 1 || Ls.J < K) && cycles(Ls) <= 0.93 * cycles(L) &&
                (Ls.N > L.N || (L.M < Ci * K && (Ci >= 128 || (Ci >= 32 && !small_layer))))) {
                L = Ls;
                xs = 1;
                s->x_off = 1 << (p - 1);
            }
        }
        if (L.N > kMaxN2D || L.segments > 8) return HIKONV_ERR_UNSUPPORTED;
        const SplitConsts sc = make_split_consts(L, p, q, xs, ws, K, L.M);
        StripProblem pr;
        pr.B = B; pr.Ci = Ci; pr.Co = Co; pr.Ho = Ho; pr.Wo = Wo; pr.N = L.N; pr.K = K; pr.J = L.J; pr.pad = pad;
        pr.moves = L.M < Ci * K;
        pr.max_moves = 1 << L.carry_bits;
        // the unrolled kernels, unless adding the upper slots while packed would overflow a slot of this layout
        pr.generic = !strip_unrolled(L.N, K, L.J);
        pr.CF = pr.generic ? 0 : move_period(L, sc, p, q, xs, ws, K, Ci, strip_packed_add(L.N, K, L.J));
        if (pr.CF == 0) {
            pr.generic = true;
            pr.CF = move_period(L, sc, p, q, xs, ws, K, Ci, false);
        }
        if (pr.CF == 0) return HIKONV_ERR_NO_FIT;                    // not even one channel's kernel rows between two moves
        for (int ks = 0; ks <= kStripMaxGroups; ++ks)
            pr.split_moves[ks] = pr.moves && !pr.generic && ks > 1 ? most_split_moves(L, sc, p, q, xs, ws, K, pr.CF, ks, strip_packed_add(L.N, K, L.J)) : 0;
        pr.requant = out.requant != 0; pr.pool = out.requant && out.pool;
        pr.xo_mult = segment_multiple(out, L.N);
        pr.sms = sm_count();
        // tune->tile > 0: rows per CTA, plus 1000 x channel lanes per CTA, 100000 x rows and 1000000 x channels per thread when
        // those are forced too
        const int tile_arg = (tune && tune->tile > 0) ? tune->tile : 0, force_ks = tile_arg / 10000000, force_tn = tile_arg / 1000000 % 10, force_tm = tile_arg / 100000 % 10;
        if ((force_tm != 0 && force_tm != 2 && force_tm != 4) || (force_tn != 0 && force_tn != 4 && force_tn != 8) ||
            force_ks == 3 || force_ks > 4) return HIKONV_ERR_UNSUPPORTED;
        const StripChoice c = choose_strips(pr, force_tm, force_tn, force_ks, tile_arg % 100000 / 1000, tile_arg % 1000);
        if (c.cost < 0) return HIKONV_ERR_UNSUPPORTED;

        StripLaunch &l = s->strip;
        StripParams &k = l.p;
        std::memset(&k, 0, sizeof(k));
        l.TM = c.TM; l.TN = c.TN; l.KS = c.KS; l.sp = L.signed_prod != 0; l.moves = pr.moves; l.generic = pr.generic; l.threads = c.threads;
        k.Ci = Ci; k.Co = Co; k.CoP = s->CoP; k.K = K; k.J = L.J; k.Ho = Ho; k.Wo = Wo; k.W = W; k.pad = pad;
        k.Hp = s->Hp; k.ap_rows = B * s->Hp;
        k.SH = ceil_div(Ho, c.TM); k.strips = B * k.SH;
        k.NSEG = c.NSEG; k.XO = c.XO; k.XB = c.XB; k.halo = c.halo; k.X = c.X; k.col_off = c.col_off; k.pitch = c.pitch;
        k.XBT = (c.NSEG - 1) * c.XO + c.pitch;
        k.TS = c.TS; k.TNX = c.TNX; k.TCO = c.TNX * c.TN; k.CK = c.CK; k.run = c.run; k.runs_per_move = c.runs_per_move; k.bar_off = c.bar_off; k.e_off = c.e_off;
        k.plane = c.plane; k.a_words = c.CK * c.plane; k.b_off = 2 * k.a_words; k.b_words = c.CK * K * L.J * kStripBPitch;
        auto magic = [](int d) -> uint32_t { return d <= 1 ? 0u : (uint32_t)((0x100000000ull + (unsigned)d - 1) / (unsigned)d); };
        k.mg_xb = magic(c.XB); k.mg_sh = magic(k.SH);
        k.S = L.S; k.SN = L.S * L.N; k.h = L.carry_bits;
        k.bias = sc.bias; k.mask_low = sc.mask_low; k.mask_high = sc.mask_high; k.slot_mask = sc.slot_mask;
        for (int m = 0; m < 8; ++m) k.slot_bias[m] = m < L.segments ? sc.seg_bias[m] : 0;
        k.up_slots = L.segments - L.N;
        k.requant = out.requant ? 1 : 0; k.shift = out.shift; k.lo = out.lo; k.hi = out.hi;
        k.pool = !pr.pool ? 0 : out.lo < 0 && out.hi > 127 ? 2 : 1;   // 2: the bytes of codes above 127 are negative
        k.out_bits = out.out_bits; k.out_signed = out.lo < 0 ? 1 : 0;
        rc = output_staging(out, Ho, Wo, c.NSEG, c.XO * L.N, &k.stage_out, &k.vec);
        if (rc != HIKONV_OK) return rc;
        k.WTP = (c.XO * L.N + 15) / 16 * 16;
        k.tile_off = (c.threads / 32 * c.TNX * c.TM * c.TN / c.KS * 2 + 3) / 4 * 4;
        const long long gx = ((long long)k.strips + c.TS - 1) / c.TS * c.NSEG;
        const int gy = ceil_div(Co, k.TCO);
        if (gx > 0x7FFFFFFFLL || gy > 65535) return HIKONV_ERR_UNSUPPORTED;
        l.grid = dim3((unsigned)gx, (unsigned)gy, 1);
        // A grid of less than one wave must spread over the SMs evenly.  The kernel is launched while the packing launch still
        // runs (programmatic dependency), and its CTAs then pile up on the SMs that are free first: 111 CTAs took 32 us one to
        // an SM and 55 to 60 us when two found room on one.  Such a grid asks for as much shared memory as lets only the
        // even share of CTAs onto an SM.
        l.smem_bytes = c.smem;
        const long long share = (c.ctas + pr.sms - 1) / pr.sms;
        if (share <= 4) l.smem_bytes = std::max(c.smem, (size_t)(kSmemPerSm / (share + 1) - 1024 + 256));

        // Words of several filters (tune->tile == -3: wherever the layer fits them, and more digits in front force parts of its tile): the slots hold the sums of the whole layer.  They are
        // the faster ones for pooled layers of few input channels whose words of pixels hold three products at best (N = 2, two words
        // per kernel row): the pool is then a thread's own pixels.  As graphs, two launches / this kernel: 3 -> 16 channels u8 x s4 on
        // 160x320 maps, 2 / 4 / 16 / 64 images 9.5 / 12.2 / 34.1 / 123.6 against 6.9 / 8.9 / 24.7 / 82.2 us; sixty-four and 256 32x32 maps
        // 6.5 / 13.1 against 5.8 / 10.0; 1 -> 16 on 1024 8x8 and 28x28 maps 5.9 / 32.3 against 4.4 / 14.7; 3 -> 32 on sixty-four 112x112 maps
        // 58.5 / 50.4; 6 -> 96 at 6 bits on thirty-two 160x320 maps 522 / 343.  Over 413 layers that the rule takes (every width it allows, 1 to
        // 6 channels, 16 to 128 filters, a million sums to 4e8) 0.63 of the time, one of them slower (3.7 %: 6 -> 39 on six 52x120 maps).
        // Below a million sums 14 of 107 were slower by more than half a per cent, up to 10 %, and what these calls take is launch and first
        // fetch, which the models of the forms do not tell apart (by their comparison 7 would still be slower): the line lies there.  The line
        // at 16 filters is older than the present tiles: 3 -> 8 and 3 -> 12 on sixteen 160x320 maps 19.5 / 17.8 and 33.9 / 19.2, on
        // sixty-four 68.1 / 57.7 and 121.6 / 62.5 would gain, too.  Nor are layers without a pool taken: over forty of them 0.64 to 1.28 of the
        // time, sums and codes alike (3 -> 16 on forty-eight 48x320 maps 30.4 / 32.6, 6 -> 39 on six 52x120 maps 10.0 / 11.1, 6 -> 36 on
        // 129 18x278 maps 110 / 71), and no line drawn between them.
        const bool own_layout = tune && (tune->N || tune->S || tune->M || tune->tile);
        const bool force_filters = tune && tune->tile <= -3 && tune->tile % 10 == -3 && !tune->N && !tune->S && !tune->M;
        if (K == kFiltersK && out.byte_inputs && out.out_bits == 8 && (!own_layout || force_filters)) {
            const double x_lo = own_xs ? -(double)(1 << (p - 1)) : 0.0, x_hi = own_xs ? (1 << (p - 1)) - 1 : (1 << p) - 1;
            const double w_lo = ws ? -(double)(1 << (q - 1)) : 0.0, w_hi = ws ? (1 << (q - 1)) - 1 : (1 << q) - 1;
            const double least = std::min(0.0, std::min(x_lo * w_hi, x_hi * w_lo));
            const double most = std::max(0.0, std::max(x_lo * w_lo, x_hi * w_hi));
            const bool fits = Ci * 9.0 * (most - least) < (double)(1 << kFiltersSlotBits);
            const bool gains = out.pool && Ci <= kFiltersMaxCi && Co >= kFiltersMinCo && L.N <= 2 && L.J >= 2 && (double)B * Ho * Wo * Co >= kFiltersMinOutputs;
            FiltersChoice fc;
            fc.cost = -1.0;
            const int digits = force_filters ? -tune->tile : 0;
            if (fits && (gains || force_filters)) fc = choose_filters(pr, {digits / 10 % 10, digits / 100 % 10, digits / 1000 % 100, digits / 100000});
            if (fc.cost >= 0 && fc.gy <= 65535 && fc.tiles <= 0x3FFFFFFF) {
                FiltersLaunch &fl = s->filt;
                FiltersParams &f = fl.p;
                std::memset(&f, 0, sizeof(f));
                f.B = B; f.Ci = Ci; f.H = H; f.W = W; f.Co = Co; f.pad = pad; f.Ho = Ho; f.Wo = Wo; f.Hp = s->Hp;
                f.SH = ceil_div(Ho, 2); f.strips = B * f.SH; f.tiles = (int)fc.tiles;
                f.NSEG = fc.NSEG; f.TQ = fc.TQ; f.TS = fc.TS; f.pos_warps = fc.pos_warps; f.groups = fc.groups;
                f.WT = fc.NW * fc.groups; f.CK = fc.CK; f.rows = fc.rows; f.PW = fc.PW; f.plane = fc.rows * fc.PW;
                f.mg_tq = magic(fc.TQ); f.mg_sh = magic(f.SH); f.mg_hp = magic(f.Hp);
                f.x_signed = own_xs; f.w_signed = ws;
                f.slot_bias = (int)(-least * Ci * 9.0);
                for (int i = 0; i < kFiltersSlots; ++i) f.bias = f.bias * (double)(1 << kFiltersSlotBits) + f.slot_bias;
                f.requant = k.requant; f.shift = out.shift; f.lo = out.lo; f.hi = out.hi; f.pool = k.pool;
                f.pair_stores = Wo % 2 == 0 && (uintptr_t)out.d_out % (out.requant ? 2 : 8) == 0 ? 1 : 0;
                fl.NW = fc.NW; fl.threads = fc.threads; fl.smem_bytes = fc.smem;
                fl.grid = dim3((unsigned)fc.gx, (unsigned)fc.gy, 1);
                const long long even = (fc.gx * fc.gy + pr.sms - 1) / pr.sms;    // spread evenly, as above
                if (even <= 4) fl.smem_bytes = std::max(fl.smem_bytes, (size_t)(kSmemPerSm / (even + 1) - 1024 + 256));
                s->filters = true;
            }
        }
        // one launch instead of two, where it is modelled to be faster (tune->tile == -1: never, -2: always)
        const bool force_small = tune && tune->tile == -2;
        if (!s->filters && !pr.generic && s->x_off == 0 && out.byte_inputs && out.out_bits == 8 && tile_arg == 0 && !(tune && tune->tile == -1)) {
            const SmallChoice sm = choose_small(pr);
            // both models brought to measured times on 66 layers (3 to 200 channels, 1 to 32 images, every layout; 8 and 16 % rms):
            // they leave out latencies of a few thousand cycles, and the packing launch takes 2.3 us and 13 us per million 16-byte
            // pieces.  Over those layers the calls took 700 us together, 719 us always in two launches, 696 us with the faster of
            // the two each time.  One launch is the faster one for little work (2x195x33x28 -> 9, 8 bits: 12.5 against 14.1 us;
            // 5x5x7x46 -> 183: 4.4 against 5.9), two from about 15 us on (9x23x16x18 -> 151, 5x5: 24.0 against 13.9)
            const double two = 4300 + 1.1 * c.cost + 0.025 * Ci * B * s->Hp * (k.XBT / 4);
            const double one = 2.4 * sm.cost - 11200 - 0.8 * std::max(0.0, sm.cost - 9800);
            if (sm.cost >= 0 && (one < two || force_small)) {
                s->one_launch = true;
                s->small_blocks = sm.XB;
                SmallLaunch &ml = s->small;
                SmallParams &mp = ml.p;
                std::memset(&mp, 0, sizeof(mp));
                mp.s = k;
                StripParams &ms = mp.s;
                ms.SH = ceil_div(Ho, kSmallTM); ms.strips = B * ms.SH;
                ms.NSEG = 1; ms.XO = ms.XB = ms.X = sm.XB; ms.halo = 0; ms.col_off = K - 1 - pad; ms.pitch = sm.pitch;
                ms.TS = sm.TS; ms.TNX = sm.TNX; ms.TCO = sm.TNX * kSmallTN;
                ms.plane = sm.rows * sm.pitch; ms.b_off = sm.Cz * ms.plane;
                ms.mg_xb = magic(sm.XB); ms.mg_sh = magic(ms.SH);
                ms.WTP = (sm.XB * L.N + 15) / 16 * 16;
                mp.B = B; mp.H = H; mp.x_signed = xs; mp.w_signed = ws; mp.Kc = L.Kc;
                mp.Cz = sm.Cz; mp.CF = pr.moves ? pr.CF : Ci + 1; mp.ks_log2 = sm.ks_log2; mp.rows = sm.rows;
                mp.col_first = -(L.J - 1) * L.N;
                mp.mg_hp = magic(s->Hp); mp.mg_xq = magic(sm.pitch / 4); mp.mg_rows = magic(sm.rows);
                mp.red_off = sm.threads / 32 * sm.TNX * kSmallTM * kSmallTN * 2;
                ms.tile_off = mp.red_off + (sm.ks_log2 > 0 ? sm.threads * kSmallTM * kSmallTN * L.N : 0);
                ml.threads = sm.threads; ml.sp = L.signed_prod != 0;
                ml.smem_bytes = sm.words * 4;
                ml.grid = dim3((unsigned)((ms.strips + sm.TS - 1) / sm.TS), (unsigned)ceil_div(Co, ms.TCO), 1u << sm.ks_log2);
                const long long even = (sm.ctas + pr.sms - 1) / pr.sms;          // spread evenly, as above
                if (even <= 4 && sm.ks_log2 == 0) ml.smem_bytes = std::max(ml.smem_bytes, (size_t)(kSmemPerSm / (even + 1) - 1024 + 256));
            }
        }
        s->XBT = k.XBT;
        s->col_first = c.halo ? K - 1 - pad - L.J * L.N : -(L.J - 1) * L.N;
        s->positions = (double)B * Ho * c.NSEG * c.XB;
    }
    s->corr_off = align_up((size_t)Ci * K * L.J * s->CoP * sizeof(uint32_t), 256);
    s->wp_bytes = s->corr_off + (s->x_off ? align_up((size_t)K * s->CoP * sizeof(int32_t), 256) : 0);
    s->ap_words = (size_t)Ci * B * s->Hp * s->XBT;
    if (s->ap_words >= 0x7FFFFFFFull || (size_t)Ci * K * L.J * s->CoP >= 0x7FFFFFFFull) return HIKONV_ERR_UNSUPPORTED;
    return HIKONV_OK;
}

// plan_layer is a function of its arguments, the SM count and the alignment of the output address, and takes longer than the
// two launches of a layer (tile choice: 60 us on average, up to 140): every thread keeps the last few plans.  No pointer is kept with them.
static int setup_layer(int B, int Ci, int H, int W, int Co, int K, int stride, int pad, int p, int q, int xs, int ws,
                       const OutputSpec &out, int algo, const hikonv_tuning_t *tune, Conv2dSetup *s) {
    struct Kept {
        int key[26];
        bool used;
        Conv2dSetup setup;
    };
    constexpr int kKept = 64;                                        // two dozen layers of a network, with room for collisions
    static thread_local Kept kept[kKept];
    const int key[26] = {B, Ci, H, W, Co, K, stride, pad, p, q, xs, ws, out.requant, out.shift, out.lo, out.hi, out.pool, out.out_bits,
                         (int)((uintptr_t)out.d_out % 16), algo, tune ? tune->N : 0, tune ? tune->S : 0, tune ? tune->M : 0,
                         tune ? tune->tile : 0, sm_count(), out.byte_inputs};
    uint32_t hash = 2166136261u;                                     // FNV-1a over the words of the key
    for (int v : key) hash = (hash ^ (uint32_t)v) * 16777619u;
    Kept &k = kept[(hash ^ (hash >> 15)) % kKept];
    if (!k.used || std::memcmp(k.key, key, sizeof(key)) != 0) {
        k.used = false;
        const int rc = plan_layer(B, Ci, H, W, Co, K, stride, pad, p, q, xs, ws, out, algo, tune, &k.setup);
        if (rc != HIKONV_OK) return rc;
        std::memcpy(k.key, key, sizeof(key));
        k.used = true;
    }
    *s = k.setup;
    return HIKONV_OK;
}

static int launch_layer(const Conv2dSetup &s, cudaStream_t st) {
    if (s.unpacked) return launch_unpacked2d(s.un, st);
    const int N = s.L.N, K = s.strip.p.K, J = s.strip.p.J;
    if (s.strip.generic) {
        switch (N) {
            case 1: return launch_strip<1, 0, 0>(s.strip, st);
            case 2: return launch_strip<2, 0, 0>(s.strip, st);
            case 3: return launch_strip<3, 0, 0>(s.strip, st);
            case 4: return launch_strip<4, 0, 0>(s.strip, st);
            default: return HIKONV_ERR_UNSUPPORTED;
        }
    }
#define HK_LAYOUT(n, k, j) if (N == n && K == k && J == j) return launch_strip<n, k, j>(s.strip, st);
    HK_LAYOUT(2, 1, 1) HK_LAYOUT(3, 1, 1) HK_LAYOUT(4, 1, 1)
    HK_LAYOUT(2, 3, 1) HK_LAYOUT(2, 3, 2) HK_LAYOUT(3, 3, 1) HK_LAYOUT(4, 3, 1)
    HK_LAYOUT(2, 5, 3) HK_LAYOUT(3, 5, 2) HK_LAYOUT(4, 5, 1) HK_LAYOUT(4, 5, 2)
#undef HK_LAYOUT
    return HIKONV_ERR_UNSUPPORTED;
}

}  // namespace hikonv

using namespace hikonv;

extern "C" size_t hikonv_conv2d_workspace_bytes(int B, int Ci, int H, int W, int Co, int K, int pad) {
    if (B < 1 || Ci < 1 || H < 1 || W < 1 || Co < 1 || K < 1 || pad < 0) return 0;
    const long long Ho = (long long)H + 2 * pad - K + 1, Wo = (long long)W + 2 * pad - K + 1;
    if (Ho < 1 || Wo < 1) return 0;
    // packed kernel rows: at most K words per (ci, kh) row (one tap per word in the comparator), Co rounded up to 4, plus one
    // int32 per channel.  The K rows of corrections of layers that run unsigned activations as signed ones fit into this:
    // with K == 1 they are that one row, and with two or more taps per word (plan_layer sees to it) the packed kernel rows leave
    // Ci K (K - J) >= K - 1 rows free
    const size_t weights = align_up((size_t)Ci * K * K * ((Co + 3) / 4 * 4) * sizeof(uint32_t), 256) +
                           align_up((size_t)((Co + 3) / 4 * 4) * sizeof(int32_t), 256);
    // packed activation rows: at most one word per output pixel plus K halo words per row (the comparator's
    // layout), rounded up to 16-byte pieces, with one more piece per row segment (segments hold >= 32 blocks)
    const size_t row_words = (size_t)(Wo + K + 3) / 4 * 4 + 16 + (size_t)(Wo + K) / 8;
    const size_t acts = (size_t)Ci * B * (size_t)(Ho + K - 1) * row_words * sizeof(uint32_t);
    return weights + align_up(acts, 256);
}

// Do the outputs of a layer on one code per byte (int32 sums or one code per byte) share memory with its inputs?  The forms in one
// launch read the inputs while CTAs that are done write outputs; in two launches the packing launch has read all of them before.
static bool writes_inputs(const void *d_x, const void *d_w, const void *d_out, int B, int Ci, int H, int W, int Co, int K, int pad, int requant, int pool) {
    if (B < 1 || Ci < 1 || H < 1 || W < 1 || Co < 1 || K < 1 || pad < 0) return false;                 // (refused by plan_layer)
    const double Ho = std::max(0.0, (double)H + 2.0 * pad - K + 1), Wo = std::max(0.0, (double)W + 2.0 * pad - K + 1);
    const double out_bytes = requant ? (double)B * Co * Ho * Wo / (pool ? 4 : 1) : 4.0 * B * Co * Ho * Wo;
    auto shares = [&](const void *d_in, double bytes) {
        const double apart = (double)(intptr_t)((uintptr_t)d_in - (uintptr_t)d_out);                     // sizes are below 2^53 or refused
        return apart < out_bytes && -apart < bytes;
    };
    return shares(d_x, (double)B * Ci * H * W) || shares(d_w, (double)Co * Ci * K * K);
}

// One layer: packing launch, then the layer kernel.  x_bits / w_bits: storage of activations and weights (8 = one code
// per byte, else dense); out_bits and pool describe the requantised output (see OutputSpec).
static int conv2d_run(const void *d_x, int x_bits, int B, int Ci, int H, int W, const void *d_w, int w_bits, int Co, int K,
                      int stride, int pad, int p, int q, int x_signed, int w_signed, void *d_out, int out_bits, int requant,
                      int shift, int lo, int hi, int pool, void *d_workspace, size_t workspace_bytes, int algo,
                      const hikonv_tuning_t *tune, void *stream) {
    if (!d_x || !d_w || !d_out) return HIKONV_ERR_INVALID_ARG;
    Conv2dSetup s;
    const OutputSpec out = {requant, shift, lo, hi, pool, out_bits, d_out,
                            x_bits == 8 && w_bits == 8 && !writes_inputs(d_x, d_w, d_out, B, Ci, H, W, Co, K, pad, requant, pool)};
    int rc = setup_layer(B, Ci, H, W, Co, K, stride, pad, p, q, x_signed ? 1 : 0, w_signed ? 1 : 0, out, algo, tune, &s);
    if (rc != HIKONV_OK) return rc;
    if (!requant && ((uintptr_t)d_out % 4) != 0) return HIKONV_ERR_INVALID_ARG;
    const size_t need = s.wp_bytes + s.ap_words * sizeof(uint32_t);
    if (!d_workspace || ((uintptr_t)d_workspace % 256) != 0 || workspace_bytes < need ||
        workspace_bytes < hikonv_conv2d_workspace_bytes(B, Ci, H, W, Co, K, pad))
        return HIKONV_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t *d_wp = (uint32_t *)d_workspace;
    uint32_t *d_ap = (uint32_t *)((char *)d_workspace + s.wp_bytes);
    int32_t *d_corr = (int32_t *)((char *)d_workspace + s.corr_off);
    if (s.unpacked) {
        s.un.p.wp = d_wp; s.un.p.ap = d_ap; s.un.p.out = d_out;
    } else {
        s.strip.p.wp = d_wp; s.strip.p.ap = d_ap; s.strip.p.out = d_out;
        s.strip.p.corr = s.x_off ? d_corr : nullptr;
    }
    const int codes = (int)((long long)B * Ci * H * W), ragged = ragged_codes(d_x, codes);        // (fewer than 2^31 codes: plan_layer)
    if (s.filters) {
        s.filt.p.x = (const int8_t *)d_x; s.filt.p.codes = codes; s.filt.p.w = (const int8_t *)d_w; s.filt.p.out = d_out;
        return launch_filters(s.filt, st);
    }
    if (s.one_launch) {
        s.small.p.x = (const int8_t *)d_x; s.small.p.ragged = ragged; s.small.p.w = (const int8_t *)d_w; s.small.p.s.out = d_out;
        return launch_small(s.small, s.L.N, st);
    }
    // a2: reversed kernel rows packed per (ci, kh, chunk); a3: activation rows packed per block; one launch
    {
        WeightPackParams wq;
        wq.w = (const int8_t *)d_w; wq.wp = d_wp; wq.Co = Co; wq.Ci = Ci; wq.K = K; wq.J = s.L.J; wq.Kc = s.L.Kc; wq.S = s.L.S;
        wq.w_signed = w_signed ? 1 : 0; wq.CoP = s.CoP; wq.w_bits = w_bits;
        wq.x_off = s.x_off; wq.corr = d_corr;
        const size_t w_warps = (size_t)ceil_div(Ci * K * s.L.J, 4) * ceil_div(s.CoP, 8);
        wq.d_cg = make_div32((uint32_t)ceil_div(s.CoP, 8));
        wq.d_j = make_div32((uint32_t)s.L.J);
        const size_t act_items = (size_t)Ci * B * s.Hp * (s.XBT / 4);              // below 2^29: ap_words is below 2^31
        const size_t act_blocks = (act_items + 255) / 256, w_blocks = (w_warps + 7) / 8;
        const size_t corr_blocks = s.x_off ? (size_t)s.CoP : 0;
        wq.w_blocks = (int)w_blocks;
        if (act_blocks + w_blocks + corr_blocks > 0x7FFFFFFFull) return HIKONV_ERR_UNSUPPORTED;
        const unsigned grid = (unsigned)(act_blocks + w_blocks + corr_blocks);
        ActPackDivs dv;
        dv.per_plane = make_div32((uint32_t)(s.Hp * (s.XBT / 4)));
        dv.b = make_div32((uint32_t)B);
        dv.xq = make_div32((uint32_t)(s.XBT / 4));
        // eight CTAs per SM where the launch has enough of them, three where it is small (see the kernel)
        const bool many = grid > 6u * (unsigned)sm_count();
        auto pack = [&](auto kern) {
            return launch_dependent(kern, dim3(grid), dim3(256), 0, st, (const int8_t *)d_x, ragged, B, Ci, H, W, s.Hp, pad, s.col_first, s.L.S,
                                    s.XBT, d_ap, (int)(w_blocks + corr_blocks), wq, x_bits, dv, (unsigned)act_items);
        };
#define HK_PACK(XSIGN, NN) rc = many ? pack(pack_operands_kernel<XSIGN, NN, 8>) : pack(pack_operands_kernel<XSIGN, NN, 3>)
        switch (s.L.N * 2 + (x_signed || s.x_off ? 1 : 0)) {
            case 2: HK_PACK(false, 1); break;
            case 3: HK_PACK(true, 1); break;
            case 4: HK_PACK(false, 2); break;
            case 5: HK_PACK(true, 2); break;
            case 6: HK_PACK(false, 3); break;
            case 7: HK_PACK(true, 3); break;
            case 8: HK_PACK(false, 4); break;
            case 9: HK_PACK(true, 4); break;
            default: return HIKONV_ERR_UNSUPPORTED;
        }
#undef HK_PACK
    }
    if (rc != HIKONV_OK) return rc;
    return launch_layer(s, st);
}

extern "C" int hikonv_conv2d_wait_timeouts(unsigned int *h_count) {
    if (!h_count) return HIKONV_ERR_INVALID_ARG;
    static int (*const counters[])(unsigned int *) = {
        strip_wait_timeouts<1, 0, 0>, strip_wait_timeouts<2, 1, 1>, strip_wait_timeouts<3, 1, 1>, strip_wait_timeouts<4, 1, 1>,
        strip_wait_timeouts<2, 3, 1>, strip_wait_timeouts<2, 3, 2>, strip_wait_timeouts<3, 3, 1>, strip_wait_timeouts<4, 3, 1>,
        strip_wait_timeouts<2, 5, 3>, strip_wait_timeouts<3, 5, 2>, strip_wait_timeouts<4, 5, 1>, strip_wait_timeouts<4, 5, 2>};
    constexpr int kDevices = 64;
    static std::mutex mutex;
    static unsigned int told[kDevices];                              // what earlier calls have reported
    *h_count = 0;
    int dev = 0;
    // all streams, the non-blocking ones too; the counters only grow, so none that comes in meanwhile is lost
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices || cudaDeviceSynchronize() != cudaSuccess) return HIKONV_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mutex);
    unsigned int total = 0;
    for (auto counter : counters) {
        unsigned int n = 0;
        const int rc = counter(&n);
        if (rc != HIKONV_OK) return rc;
        total += n;
    }
    *h_count = total - told[dev];
    told[dev] = total;
    return HIKONV_OK;
}

extern "C" int hikonv_conv2d_wait_check(long long cycles, void *stream) {
    if (cycles < 0 || cycles > kWaitCycles) return HIKONV_ERR_INVALID_ARG;
    return launch_wait_check(cycles, (cudaStream_t)stream);
}

extern "C" int hikonv_conv2d(const int8_t *d_x, int B, int Ci, int H, int W, const int8_t *d_w, int Co, int K, int stride,
                             int pad, int p, int q, int x_signed, int w_signed, void *d_out, int requant, int shift, int lo,
                             int hi, void *d_workspace, size_t workspace_bytes, int algo, const hikonv_tuning_t *tune,
                             void *stream) {
    return conv2d_run(d_x, 8, B, Ci, H, W, d_w, 8, Co, K, stride, pad, p, q, x_signed, w_signed, d_out, 8, requant, shift, lo, hi, 0,
                      d_workspace, workspace_bytes, algo, tune, stream);
}

static bool storage_bits_ok(int store_bits, int code_bits) {
    return store_bits == 8 || (store_bits == code_bits && (code_bits == 1 || code_bits == 2 || code_bits == 4));
}

extern "C" int hikonv_conv2d_dense(const void *d_x, int x_store_bits, int B, int Ci, int H, int W, const void *d_w,
                                   int w_store_bits, int Co, int K, int stride, int pad, int p, int q, int x_signed,
                                   int w_signed, void *d_out, int out_store_bits, int requant, int shift, int lo, int hi,
                                   int pool, void *d_workspace, size_t workspace_bytes, int algo,
                                   const hikonv_tuning_t *tune, void *stream) {
    if (validate_codes(p, q) != HIKONV_OK) return HIKONV_ERR_INVALID_ARG;
    if (!storage_bits_ok(x_store_bits, p) || !storage_bits_ok(w_store_bits, q)) return HIKONV_ERR_UNSUPPORTED;
    if (!requant && out_store_bits != 32) return HIKONV_ERR_INVALID_ARG;
    if (requant && out_store_bits != 8 && out_store_bits != 4 && out_store_bits != 2 && out_store_bits != 1)
        return HIKONV_ERR_INVALID_ARG;
    return conv2d_run(d_x, x_store_bits, B, Ci, H, W, d_w, w_store_bits, Co, K, stride, pad, p, q, x_signed, w_signed, d_out,
                      requant ? out_store_bits : 8, requant, shift, lo, hi, pool, d_workspace, workspace_bytes, algo, tune, stream);
}

// Times the layer with the library's own choice and with every tile of one thread group (rows x channels per thread x channel lanes x
// rows per CTA), `batch` launches between two events, best of `repeats`; the result of every launch is the layer's output.
extern "C" int hikonv_conv2d_tune(const void *d_x, int x_store_bits, int B, int Ci, int H, int W, const void *d_w,
                                  int w_store_bits, int Co, int K, int stride, int pad, int p, int q, int x_signed,
                                  int w_signed, void *d_out, int out_store_bits, int requant, int shift, int lo, int hi,
                                  int pool, void *d_workspace, size_t workspace_bytes, int algo, int repeats, int *h_tile,
                                  double *h_us, double *h_default_us, void *stream) {
    if (!h_tile || repeats < 1 || repeats > 100) return HIKONV_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t e0, e1;
    HIKONV_CUDA_TRY(cudaEventCreate(&e0));
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return HIKONV_ERR_CUDA;
    }
    constexpr int kBatch = 4;
    // best time in microseconds per launch with this tuning record; negative: the library refused it; rc_cuda set on a CUDA error
    int rc_cuda = HIKONV_OK;
    auto run = [&](const hikonv_tuning_t *tune) {
        return hikonv_conv2d_dense(d_x, x_store_bits, B, Ci, H, W, d_w, w_store_bits, Co, K, stride, pad, p, q, x_signed, w_signed,
                                   d_out, out_store_bits, requant, shift, lo, hi, pool, d_workspace, workspace_bytes, algo, tune, stream);
    };
    auto time_of = [&](const hikonv_tuning_t *tune, double give_up_above) -> double {
        float ms = 0.0f;
        if (cudaEventRecord(e0, st) != cudaSuccess) { rc_cuda = HIKONV_ERR_CUDA; return -1.0; }
        const int rc = run(tune);
        if (rc != HIKONV_OK) {
            if (rc == HIKONV_ERR_CUDA) rc_cuda = rc;
            return -1.0;
        }
        if (cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
            cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) { rc_cuda = HIKONV_ERR_CUDA; return -1.0; }
        if (ms * 1e3 > give_up_above) return ms * 1e3;               // a first launch this slow cannot win
        double best = 1e30;
        for (int rep = 0; rep < repeats; ++rep) {
            if (cudaEventRecord(e0, st) != cudaSuccess) { rc_cuda = HIKONV_ERR_CUDA; return -1.0; }
            for (int k = 0; k < kBatch; ++k)
                if (run(tune) != HIKONV_OK) { rc_cuda = HIKONV_ERR_CUDA; return -1.0; }
            if (cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
                cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) { rc_cuda = HIKONV_ERR_CUDA; return -1.0; }
            best = std::min(best, (double)ms * 1e3 / kBatch);
        }
        return best;
    };
    int rc = run(nullptr);                                            // argument errors surface here, before any timing
    double base = -1.0;
    if (rc == HIKONV_OK) {
        base = time_of(nullptr, 1e30);
        if (base < 0.0) rc = rc_cuda != HIKONV_OK ? rc_cuda : HIKONV_ERR_CUDA;
    }
    double best = base;
    int best_tile = 0;
    if (rc == HIKONV_OK) {
        const long long rows = (long long)B * ((long long)H + 2 * pad - K + 1);
        const bool packed = algo == HIKONV_ALGO_PACKED32;
        for (int shape = packed ? 3 : 1; shape >= 1 && rc_cuda == HIKONV_OK; --shape)
            for (int tnx = 1; tnx <= 8 && rc_cuda == HIKONV_OK; tnx *= 2)
                for (int tr = 1; tr <= 48 && tr <= rows + 3 && rc_cuda == HIKONV_OK; ++tr) {
                    // packed: 4 x 8, 2 x 8 and 2 x 4 rows x channels per thread, whole strips of rows
                    const int tm = shape == 3 ? 4 : 2, tn = shape >= 2 ? 8 : 4;
                    if (packed && tr % tm != 0) continue;
                    hikonv_tuning_t tune;
                    std::memset(&tune, 0, sizeof(tune));
                    tune.tile = packed ? tr + 1000 * tnx + 100000 * tm + 1000000 * tn : tr + 1000 * tnx;
                    const double t = time_of(&tune, 2.0 * best);
                    if (t >= 0.0 && t < best) { best = t; best_tile = tune.tile; }
                }
        if (rc_cuda != HIKONV_OK) rc = rc_cuda;
    }
    if (rc == HIKONV_OK && best_tile != 0 && best > 0.97 * base) { best = base; best_tile = 0; }   // not worth forcing
    if (rc == HIKONV_OK && best_tile != 0) {
        hikonv_tuning_t tune;                                          // leave d_out written by a complete, untimed launch
        std::memset(&tune, 0, sizeof(tune));
        tune.tile = best_tile;
        rc = run(&tune);
    } else if (rc == HIKONV_OK) {
        rc = run(nullptr);
    }
    if (rc == HIKONV_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = HIKONV_ERR_CUDA;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc != HIKONV_OK) return rc;
    *h_tile = best_tile;
    if (h_us) *h_us = best;
    if (h_default_us) *h_default_us = base;
    return HIKONV_OK;
}

// ---- scratch that needs no allocation: a fixed buffer inside the library image, one copy per GPU
static __device__ __align__(256) unsigned char g_static_scratch[HIKONV_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void *g_scratch_ptr[kMaxDevices] = {nullptr};

// Is `ptr` device memory of GPU `dev`?  (A query of the pointer's attributes; nothing is allocated.)
bool on_device(const void *ptr, int dev) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged) && attr.device == dev;
}

// Device address of g_static_scratch on the current device.  In host code the array's name is only
// a handle, so the address is asked for once per device and cached.  The buffer of the CURRENT device is
// used, so the operands must live there: a buffer of one GPU must not reach kernels that run on another.
int static_scratch_address(void **out, const void *d_x, const void *d_out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return HIKONV_ERR_CUDA;
    if (!d_x || !d_out || !on_device(d_x, dev) || !on_device(d_out, dev)) return HIKONV_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_ptr[dev]) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) return HIKONV_ERR_CUDA;
        g_scratch_ptr[dev] = ptr;
    }
    *out = g_scratch_ptr[dev];
    return HIKONV_OK;
}
}  // namespace

extern "C" int hikonv_conv2d_static_scratch(const int8_t *d_x, int B, int Ci, int H, int W, const int8_t *d_w, int Co, int K,
                                            int stride, int pad, int p, int q, int x_signed, int w_signed, void *d_out,
                                            int requant, int shift, int lo, int hi, int algo, const hikonv_tuning_t *tune,
                                            void *stream) {
    const size_t need = hikonv_conv2d_workspace_bytes(B, Ci, H, W, Co, K, pad);
    if (need == 0) return HIKONV_ERR_INVALID_ARG;
    if (need > (size_t)HIKONV_STATIC_SCRATCH_BYTES) return HIKONV_ERR_TOO_LARGE;
    void *scratch = nullptr;
    const int rc = static_scratch_address(&scratch, d_x, d_out);
    if (rc != HIKONV_OK) return rc;
    // the packing kernels write every word the layer kernel reads, so stale contents are harmless
    return hikonv_conv2d(d_x, B, Ci, H, W, d_w, Co, K, stride, pad, p, q, x_signed, w_signed, d_out, requant, shift, lo, hi,
                         scratch, (size_t)HIKONV_STATIC_SCRATCH_BYTES, algo, tune, stream);
}

extern "C" size_t hikonv_conv2d_host_workspace_bytes(int B, int Ci, int H, int W, int Co, int K, int pad, int requant) {
    if (B < 1 || Ci < 1 || H < 1 || W < 1 || Co < 1 || K < 1 || pad < 0) return 0;
    const long long Ho = H + 2 * pad - K + 1, Wo = W + 2 * pad - K + 1;
    if (Ho < 1 || Wo < 1) return 0;
    const size_t out_bytes = (size_t)B * Co * Ho * Wo * (requant ? 1 : 4);
    return align_up((size_t)B * Ci * H * W, 256) + align_up((size_t)Co * Ci * K * K, 256) + align_up(out_bytes, 256) +
           hikonv_conv2d_workspace_bytes(B, Ci, H, W, Co, K, pad);
}

extern "C" int hikonv_conv2d_host(const int8_t *h_x, int B, int Ci, int H, int W, const int8_t *h_w, int Co, int K, int stride,
                                  int pad, int p, int q, int x_signed, int w_signed, void *h_out, int requant, int shift, int lo,
                                  int hi, void *d_workspace, size_t workspace_bytes, int algo, const hikonv_tuning_t *tune,
                                  void *stream) {
    if (!h_x || !h_w || !h_out) return HIKONV_ERR_INVALID_ARG;
    const size_t need = hikonv_conv2d_host_workspace_bytes(B, Ci, H, W, Co, K, pad, requant);
    if (need == 0) return HIKONV_ERR_INVALID_ARG;
    if (!d_workspace || ((uintptr_t)d_workspace % 256) != 0 || workspace_bytes < need) return HIKONV_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t x_bytes = (size_t)B * Ci * H * W, w_bytes = (size_t)Co * Ci * K * K;
    const size_t Ho = H + 2 * pad - K + 1, Wo = W + 2 * pad - K + 1;
    const size_t out_bytes = (size_t)B * Co * Ho * Wo * (requant ? 1 : 4);
    int8_t *d_x = (int8_t *)d_workspace;
    int8_t *d_w = d_x + align_up(x_bytes, 256);
    int8_t *d_out = d_w + align_up(w_bytes, 256);
    int8_t *d_ws = d_out + align_up(out_bytes, 256);
    HIKONV_CUDA_TRY(cudaMemcpyAsync(d_x, h_x, x_bytes, cudaMemcpyHostToDevice, st));
    HIKONV_CUDA_TRY(cudaMemcpyAsync(d_w, h_w, w_bytes, cudaMemcpyHostToDevice, st));
    const int rc = hikonv_conv2d(d_x, B, Ci, H, W, d_w, Co, K, stride, pad, p, q, x_signed, w_signed, d_out, requant, shift, lo,
                                 hi, d_ws, hikonv_conv2d_workspace_bytes(B, Ci, H, W, Co, K, pad), algo, tune, st);
    if (rc != HIKONV_OK) return rc;
    HIKONV_CUDA_TRY(cudaMemcpyAsync(h_out, d_out, out_bytes, cudaMemcpyDeviceToHost, st));
    return HIKONV_OK;
}

extern "C" int hikonv_maxpool2x2_i8(const int8_t *d_in, int B, int C, int H, int W, int is_signed, int8_t *d_out, void *stream) {
    if (!d_in || !d_out || B < 1 || C < 1 || H < 1 || W < 1) return HIKONV_ERR_INVALID_ARG;
    const long long total = (long long)B * C * (H / 2) * (W / 2);
    if (total == 0) return HIKONV_OK;
    if ((double)B * C >= 2147483647.0) return HIKONV_ERR_UNSUPPORTED;
    const long long cap = (long long)sm_count() * 32;
    const cudaStream_t pst = (cudaStream_t)stream;
    if (W % 16 == 0 && ((uintptr_t)d_in % 16) == 0 && ((uintptr_t)d_out % 8) == 0) {
        const long long items = total / 8;
        const unsigned grid = (unsigned)std::min((items + 255) / 256, cap);
        if (is_signed) return launch_dependent(maxpool2x2_vec_kernel<true, 16>, dim3(grid), dim3(256), 0, pst, d_in, items, H, W, d_out);
        return launch_dependent(maxpool2x2_vec_kernel<false, 16>, dim3(grid), dim3(256), 0, pst, d_in, items, H, W, d_out);
    }
    if (W % 8 == 0 && ((uintptr_t)d_in % 8) == 0 && ((uintptr_t)d_out % 4) == 0) {
        const long long items = total / 4;
        const unsigned grid = (unsigned)std::min((items + 255) / 256, cap);
        if (is_signed) return launch_dependent(maxpool2x2_vec_kernel<true, 8>, dim3(grid), dim3(256), 0, pst, d_in, items, H, W, d_out);
        return launch_dependent(maxpool2x2_vec_kernel<false, 8>, dim3(grid), dim3(256), 0, pst, d_in, items, H, W, d_out);
    }
    long long blocks = (total + 255) / 256;
    if (blocks > cap) blocks = cap;
    return launch_plain(maxpool2x2_kernel, dim3((unsigned)blocks), dim3(256), 0, (cudaStream_t)stream, d_in, B * C, H, W,
                        is_signed ? 1 : 0, d_out);
}

extern "C" int hikonv_conv2d_layout(int B, int Ci, int H, int W, int Co, int K, int pad, int p, int q, int x_signed,
                                    int w_signed, const hikonv_tuning_t *tune, hikonv_layout_t *out, int *x_shift) {
    if (!out) return HIKONV_ERR_INVALID_ARG;
    Conv2dSetup s;
    const OutputSpec sums = {0, 0, 0, 0, 0, 8, nullptr, 0};
    const int rc = setup_layer(B, Ci, H, W, Co, K, 1, pad, p, q, x_signed ? 1 : 0, w_signed ? 1 : 0, sums, HIKONV_ALGO_PACKED32, tune, &s);
    if (rc != HIKONV_OK) return rc;
    *out = s.L;
    if (x_shift) *x_shift = s.x_off;
    return HIKONV_OK;
}

extern "C" int hikonv_conv2d_launches(int B, int Ci, int H, int W, int Co, int K, int pad, int p, int q, int x_signed, int w_signed,
                                      int requant, int pool, const hikonv_tuning_t *tune, int *launches, int *cluster) {
    if (!launches) return HIKONV_ERR_INVALID_ARG;
    Conv2dSetup s;
    const OutputSpec out = {requant ? 1 : 0, 0, 0, 0, pool ? 1 : 0, 8, nullptr, 1};
    const int rc = setup_layer(B, Ci, H, W, Co, K, 1, pad, p, q, x_signed ? 1 : 0, w_signed ? 1 : 0, out, HIKONV_ALGO_PACKED32, tune, &s);
    if (rc != HIKONV_OK) return rc;
    *launches = s.one_launch || s.filters ? 1 : 2;
    if (cluster) *cluster = s.filters ? 1 : s.one_launch ? (int)s.small.grid.z : 0;
    return HIKONV_OK;
}

extern "C" int hikonv_conv2d_form(int B, int Ci, int H, int W, int Co, int K, int pad, int p, int q, int x_signed, int w_signed, int requant,
                                  int pool, int algo, const hikonv_tuning_t *tune, hikonv_conv2d_form_t *form) {
    if (!form) return HIKONV_ERR_INVALID_ARG;
    Conv2dSetup s;
    const OutputSpec out = {requant ? 1 : 0, 0, 0, 0, pool ? 1 : 0, 8, nullptr, 1};
    const int rc = setup_layer(B, Ci, H, W, Co, K, 1, pad, p, q, x_signed ? 1 : 0, w_signed ? 1 : 0, out, algo, tune, &s);
    if (rc != HIKONV_OK) return rc;
    std::memset(form, 0, sizeof(*form));
    const double rows = (double)B * (H + 2 * pad - K + 1), row = W + 2 * pad - K + 1, pairs = (double)Ci * K;    // (input channel, kernel row) pairs
    if (!s.unpacked && s.filters) {
        const FiltersParams &f = s.filt.p;
        form->form = HIKONV_FORM_FILTERS;
        form->launches = 1;
        form->words = s.filt.NW; form->groups = f.groups; form->step_channels = f.CK;
        form->ctas = (int)s.filt.grid.x; form->tiles = f.tiles; form->segments = f.NSEG;
        form->double_multiplies = rows * row * ceil_div(Co, kFiltersSlots) * pairs * K;
        return HIKONV_OK;
    }
    form->form = s.unpacked ? HIKONV_FORM_UNPACKED : s.one_launch ? HIKONV_FORM_ONE_LAUNCH : HIKONV_FORM_TWO_LAUNCHES;
    form->launches = form->form == HIKONV_FORM_ONE_LAUNCH ? 1 : 2;
    form->cluster = form->form == HIKONV_FORM_ONE_LAUNCH ? (int)s.small.grid.z : 0;
    form->multiplies = (form->form == HIKONV_FORM_ONE_LAUNCH ? rows * s.small_blocks : s.positions) * Co * pairs * s.L.J;
    return HIKONV_OK;
}

extern "C" double hikonv_conv2d_multiplies(int B, int Ci, int H, int W, int Co, int K, int pad, int p, int q, int x_signed,
                                           int w_signed, int algo, const hikonv_tuning_t *tune) {
    Conv2dSetup s;
    const OutputSpec sums = {0, 0, 0, 0, 0, 8, nullptr, 0};
    if (setup_layer(B, Ci, H, W, Co, K, 1, pad, p, q, x_signed ? 1 : 0, w_signed ? 1 : 0, sums, algo, tune, &s) != HIKONV_OK) return 0.0;
    // one multiply per position, channel pair and (kh, j): halo positions included, idle threads not
    return s.positions * (double)Co * Ci * K * s.L.J;
}
