// The packed layer kernel.  A layer is computed as row-wise packed 1-D convolutions (Theorem 3) whose products are summed
// over input channels and kernel rows in 64-bit packed accumulators before the split (Eq. 23).
//
// Work decomposition.  Group x of an output row is N neighbouring columns; its packed input word A_x (Eq. 5) gives
//     Q_x = bias + sum_{ci, kh, j} A[ci][row + kh][x - j] * Bw[ci][kh][j]
// whose slots m < N belong to group x and slots m >= N to group x + 1 (Theorem 2).  A thread owns a STRIP of TM
// neighbouring output rows at one group and TN output channels: the TM + K - 1 activation words of a channel serve all K
// kernel rows (a 4 x 4 tile loads 6 words and three 16-byte weight pieces for 48 multiplies; with four positions of one row
// per thread it loaded 12), and all index arithmetic is done for one position instead of TM.  Lanes run along the row, so the
// group in front of a lane's is in the lane before it, whatever the row of the strip.
//
// A CTA computes TS consecutive strips (of one or several images) of one row segment times TCO channels.  Packed activation
// rows and kernel rows are streamed in stages of CK input channels with asynchronous copies into double-buffered shared memory.
//
// Thread groups.  A layer of few strips leaves schedulers with one or two warps, which cannot hide each other's latencies, or SMs
// with nothing.  There KS groups of threads work on one tile, each on its share of a stage's input channels; the packed sums (and
// second accumulators) are added in shared memory, and every group splits and stores TN / KS of the channels.  Each group has the
// prologue and the moves to itself, so this is for layers that lack warps, by the cost model's estimate: 32 images 128x7x7 -> 256
// 30.9 -> 23.9 us, 1x175x15x62 -> 57 5x5 104 -> 35 us (four groups), 4x128x28x28 -> 128 31.3 -> 24.3 us; but 56x56x64 (four
// warps per scheduler without) 86.6 -> 100 us.
//
// Split.  Every slot starts at a bias that makes its running sum non-negative, so slots never borrow from each other (this
// replaces the sign-borrow increment of Eq. 29).  After CF input channels a slot could overflow; the bits of every slot above
// its low h then move to a SECOND packed accumulator with the same layout,
//     E += (Q >> h) & mask_high;      Q = (Q & mask_low) | bias,
// which takes 2^h such moves.  At the end the words above the N low slots travel to the next lane still packed and are added
// there (packed_add; where the slots do not have the room for that, as separate fields), the N slots are read by shift and
// mask, value m = 2^h E_m + Q_m - (moves + 1) (bias_m + bias_{m + N}).
//
// What bounds it: the multiplier's pipe and the instruction issue around it.  A warp-wide 32x32->64 multiply-add holds its
// scheduler for 4.1 cycles in a loop of nothing else; in this loop a channel of a 4 x 8 tile (96 of them, 34 other
// instructions) takes 473 cycles, of a 2 x 8 tile with moves (48 and 52) 285.  Three CTAs per SM, operand rows in registers
// across channels or a compile-time distance between channels (no pointer arithmetic left) changed neither.
// Measured against the kernel before it (four positions of one row per thread, one halo word per row, run-time loops for 5x5),
// packing launch included: 32x64x56x56 -> 64 s4 93.3 -> 84.6 us, 64x256x14x14 -> 256 u4 x s4 211 -> 160 us (205 with the new
// packing launch alone), 8x48x37x53 -> 40 s8 32.4 -> 26.3 us, 16x24x45x61 -> 40 5x5 2-bit 70.6 -> 30.0 us, the compact CNN
// (batch 64) 605 -> 475 us.
#pragma once

#include <type_traits>

#include "hikonv_cuda.cuh"
#include "hikonv_conv2d_strip.h"
#include "hikonv_conv2d_util.cuh"

namespace hikonv {

// Threads of this file's kernels whose wait for a stage ran out (one counter per file, which only grows).
static __device__ unsigned int strip_timeouts;

template <int N, int KT, int JT>
constexpr bool kStripPackedAdd = strip_packed_add(N, KT, JT);

// N: pixels per word; KT, JT: kernel size and words per kernel row (0: run-time bounds); TM x TN: rows x channels per thread;
// SP: signed product; HASE: with second accumulators; KS: thread
// groups that share the input channels of a tile.
template <int N, int KT, int JT, int TM, int TN, bool SP, bool HASE, int KS>
__global__ void __launch_bounds__(kStripThreads, 2) conv2d_strip_kernel(const __grid_constant__ StripParams p) {
    constexpr bool PACKED_ADD = kStripPackedAdd<N, KT, JT>;
    constexpr bool UP = N > 1 && KT != 1;                       // some products have slots above the N low ones
    constexpr int ROWS = KT > 0 ? TM + KT - 1 : TM;            // activation rows a thread points at
    extern __shared__ __align__(16) uint32_t smem[];
    grid_dependency_release();

    const int tid = threadIdx.x, nthreads = blockDim.x, lane = tid & 31;
    const int warp = tid >> 5;
    const int group_threads = nthreads / KS, group = KS > 1 ? warp / ((nthreads / KS) >> 5) : 0, gtid = tid - group * group_threads;
    constexpr int TE = TN / KS;                                // channels that a thread finishes: TE group ..
    const int tnx_log2 = 31 - __clz(p.TNX);                    // TNX is a power of two
    const int tn = gtid & (p.TNX - 1);
    const int strip_tile = p.NSEG > 1 ? (int)(blockIdx.x / (unsigned)p.NSEG) : (int)blockIdx.x;
    const int seg = (int)blockIdx.x - strip_tile * p.NSEG;
    const int g0 = strip_tile * p.TS;                          // first strip
    const int b0 = g0 / p.SH, s0 = g0 - b0 * p.SH;
    const int TSe = min(p.TS, p.strips - g0);
    const int co0 = blockIdx.y * p.TCO;
    const int K = KT > 0 ? KT : p.K, J = JT > 0 ? JT : p.J;

    // staged rows: from the first row of the first strip to the last row of the last one (rows past the last image do not exist)
    const int r0 = b0 * p.Hp + s0 * TM;
    const int tl = s0 + TSe - 1, dbl = fast_div(tl, p.mg_sh);
    const int NR = min(dbl * p.Hp + (tl - dbl * p.SH) * TM - s0 * TM + TM + K - 1, p.ap_rows - r0);

    // this thread's strip and group (an idle thread works on position 0; its results are dropped)
    const int pos = gtid >> tnx_log2, pos_ok = pos < TSe * p.XB, pc = pos_ok ? pos : 0;
    const int sl = fast_div(pc, p.mg_xb), xb = pc - sl * p.XB;
    const int db = fast_div(s0 + sl, p.mg_sh), s_img = s0 + sl - db * p.SH;
    int a_off[ROWS];                                           // word of row r, j = 0 in a channel's plane
#pragma unroll
    for (int r = 0; r < ROWS; ++r) a_off[r] = (db * p.Hp + (s_img - s0) * TM + r) * p.pitch + xb + J - 1;

    // Second accumulators: in shared memory, at an odd pitch of 8-byte entries per thread, so that the lanes of a warp fall into
    // different banks and every access has an immediate offset.  They are touched once in CF channels; in registers they would
    // leave no room for 32 accumulators (and with 16 they were no faster).
    uint64_t acc[TM][TN];
    uint2 *es = reinterpret_cast<uint2 *>(smem + p.e_off) + tid * strip_e_pitch(TM, TN);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int t = 0; t < TN; ++t) {
            acc[i][t] = p.bias;
            if constexpr (HASE) es[i * TN + t] = make_uint2(0u, 0u);
        }
    auto move_upper_bits = [&]() {
        if constexpr (HASE) {
            const uint32_t mh_lo = (uint32_t)p.mask_high, mh_hi = (uint32_t)(p.mask_high >> 32);
            const uint32_t ml_lo = (uint32_t)p.mask_low, ml_hi = (uint32_t)(p.mask_low >> 32);
            const uint32_t b_lo = (uint32_t)p.bias, b_hi = (uint32_t)(p.bias >> 32);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int t = 0; t < TN; ++t) {
                    const uint32_t q_lo = (uint32_t)acc[i][t], q_hi = (uint32_t)(acc[i][t] >> 32);
                    const uint32_t h_lo = __funnelshift_r(q_lo, q_hi, p.h) & mh_lo, h_hi = (q_hi >> p.h) & mh_hi;
                    uint2 e = es[i * TN + t];
                    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+r"(e.x), "+r"(e.y) : "r"(h_lo), "r"(h_hi));
                    es[i * TN + t] = e;
                    acc[i][t] = ((uint64_t)((q_hi & ml_hi) | b_hi) << 32) | ((q_lo & ml_lo) | b_lo);
                }
        }
    };

    // Asynchronous fetch of the next ckn input channels.  Activations by bulk copies dealt to the warps (with warp 0 issuing all
    // of them the others waited for it): the staged rows of a channel are contiguous when rows are uncut, else each row is a
    // copy.  Kernel words, short pieces at a constant pitch, by 16-byte copies of the threads (what lies behind the last channel
    // keeps old contents: the accumulators there are never stored).
    uint32_t *const Bs = smem + p.b_off;
    const uint32_t bar0 = smem_address(smem + p.bar_off);
    const int KJ = K * J, nwarps = nthreads >> 5;
    const uint32_t row_bytes = 4u * (uint32_t)p.pitch, ch_bytes = NR * row_bytes;
    const size_t ap_plane = (size_t)p.ap_rows * p.XBT;
    const int tco4_log2 = 29 - __clz(p.TCO), b_row = tid >> tco4_log2, b_col = 4 * (tid & (p.TCO / 4 - 1));   // TCO / 4 is a power of two
    const int b_step = nthreads >> tco4_log2, b_rows = co0 + b_col < p.CoP ? 0x7FFFFFFF : 0;
    const uint32_t *a_next = p.ap + (size_t)r0 * p.XBT + seg * p.XO + (p.NSEG == 1 ? warp * ap_plane : 0);   // of the stage to fetch next
    const uint32_t *b_next = p.wp + (size_t)b_row * p.CoP + co0 + b_col;
    const size_t a_stage = p.CK * ap_plane, b_stage = (size_t)p.CK * KJ * p.CoP;
    const uint32_t a_dst0 = smem_address(smem), b_dst0 = smem_address(Bs + b_row * kStripBPitch + b_col);
    auto fetch = [&](int ckn, int stage) {
        const uint32_t bar = bar0 + 8u * stage, a_dst = a_dst0 + 4u * stage * p.a_words;
        if (tid == 0) mbarrier_arrive_expect(bar, ckn * ch_bytes);
        if (p.NSEG == 1) {
            if (lane == 0) {
                if (warp < ckn) bulk_copy(a_dst + 4u * warp * p.plane, a_next, ch_bytes, bar);
                for (int c = warp + nwarps; c < ckn; c += nwarps)
                    bulk_copy(a_dst + 4u * c * p.plane, a_next + (size_t)(c - warp) * ap_plane, ch_bytes, bar);
            }
        } else {
            const float inv_nr = 1.0f / (float)NR;
            for (int q = lane * nwarps + warp; q < ckn * NR; q += nthreads) {
                const int c = small_div(q, NR, inv_nr), r = q - c * NR;
                bulk_copy(a_dst + 4u * c * p.plane + r * row_bytes, a_next + c * ap_plane + (size_t)r * p.XBT, row_bytes, bar);
            }
        }
        const int rows = min(ckn * KJ, b_rows);
        const uint32_t b_dst = b_dst0 + 4u * stage * p.b_words;
        if (b_row < rows) cp_async_16_at(b_dst, b_next);
        for (int k = b_row + b_step, n = 1; k < rows; k += b_step, ++n)
            cp_async_16_at(b_dst + n * (4u * kStripBPitch) * b_step, b_next + (size_t)(n * b_step) * p.CoP);
        cp_async_commit();
        a_next += a_stage;
        b_next += b_stage;
    };
    if (tid == 0) {
        mbarrier_init(bar0, 1);
        mbarrier_init(bar0 + 8, 1);
        mbarrier_init_fence();
    }
    __syncthreads();
    grid_dependency_wait();                                    // everything above touched no global memory
    fetch(min(p.CK, p.Ci), 0);

    // one input channel: activations from word a_ch of shared memory on, kernel words from word b_ch on (the same for the CTA)
    const int b_tn = tn * TN;
    auto channel = [&](int a_ch, int b_ch) {
        if constexpr (KT > 0) {
            uint32_t a[ROWS][JT];
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
#pragma unroll
                for (int j = 0; j < JT; ++j) a[r][j] = smem[a_ch + a_off[r] - j];
#pragma unroll
            for (int kh = 0; kh < KT; ++kh)
#pragma unroll
                for (int j = 0; j < JT; ++j) {
                    uint32_t b[TN];
#pragma unroll
                    for (int t = 0; t < TN; t += 4) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(smem + b_ch + b_tn + (kh * JT + j) * kStripBPitch + t);
                        b[t] = v.x; b[t + 1] = v.y; b[t + 2] = v.z; b[t + 3] = v.w;
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int t = 0; t < TN; ++t) mad_wide<SP>(acc[i][t], a[i + kh][j], b[t]);
                }
        } else {
            for (int kh = 0; kh < K; ++kh)
                for (int j = 0; j < J; ++j, b_ch += kStripBPitch) {
                    uint32_t a[TM], b[TN];
#pragma unroll
                    for (int i = 0; i < TM; ++i) a[i] = smem[a_ch + a_off[i] + kh * p.pitch - j];
#pragma unroll
                    for (int t = 0; t < TN; t += 4) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(smem + b_ch + b_tn + t);
                        b[t] = v.x; b[t + 1] = v.y; b[t + 2] = v.z; b[t + 3] = v.w;
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int t = 0; t < TN; ++t) mad_wide<SP>(acc[i][t], a[i], b[t]);
                }
        }
    };
    // a run of input channels between two possible moves: the whole stage, or CF channels of it
    const int run = HASE ? p.run : p.CK;
    int moves = 0, runs_left = p.runs_per_move;
    uint32_t parity = 0;                                       // of this stage's barrier; both buffers' barriers flip every second stage
    int stage = 0;
    for (int ci0 = 0; ci0 < p.Ci; ci0 += p.CK, stage ^= 1) {
        const int ckn = min(p.CK, p.Ci - ci0);
        // the groups' shares of a stage (the last ones' may be shorter; moves happen at the same places in all)
        const int share = (ckn + KS - 1) / KS, own = min(ckn - group * share, share);
        // this stage has landed, and the previous one is fully consumed.  Were a wait ever to run out, the CTA would count it, wait
        // for its copies once more (those of this stage are all that can be in flight) and leave its outputs unwritten
        const bool landed = mbarrier_wait(bar0 + 8u * stage, parity);
        cp_async_wait_all();
        if (__syncthreads_or(!landed)) {
            if (!landed) atomicAdd(&strip_timeouts, 1u);
            mbarrier_wait(bar0 + 8u * stage, parity);
            return;
        }
        parity ^= (uint32_t)stage;
        if (ci0 + p.CK < p.Ci) fetch(min(p.CK, p.Ci - ci0 - p.CK), stage ^ 1);
        int a_ch = stage * p.a_words, b_ch = p.b_off + stage * p.b_words;
        if constexpr (KS > 1) {
            a_ch += group * share * p.plane;
            b_ch += group * share * KJ * kStripBPitch;
        }
        for (int c = 0; c < share; c += run) {
            const int n = HASE ? min(run, own - c) : own;
#pragma unroll 2
            for (int u = 0; u < n; ++u, a_ch += p.plane, b_ch += KJ * kStripBPitch) channel(a_ch, b_ch);
            if constexpr (HASE) {
                if (--runs_left == 0 && (c + run < share || ci0 + p.CK < p.Ci)) {  // none is needed after the last channel
                    move_upper_bits();
                    ++moves;
                    runs_left = p.runs_per_move;
                }
            }
        }
    }

    // ---- several groups: each finishes a share of a tile's channels, summed through shared memory.  Of the KS biases in a sum all
    // but one are taken off; the bits above the low h have all moved before, so no slot overflows
    uint2 *const xch0 = reinterpret_cast<uint2 *>(smem);
    uint64_t fin[TM][TE];
    __syncthreads();
    if constexpr (KS > 1) {
        if constexpr (HASE) {
            move_upper_bits();
            ++moves;
        }
        uint2 *const sums = xch0 + (nthreads >> 5) * p.TNX * (TM * TE);
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int t = 0; t < TN; ++t) sums[(i * TN + t) * nthreads + tid] = make_uint2((uint32_t)acc[i][t], (uint32_t)(acc[i][t] >> 32));
        __syncthreads();
        const uint2 *from = sums + group * TE * nthreads + gtid;
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int t = 0; t < TE; ++t) {
                uint64_t v = (uint64_t)(1 - KS) * p.bias;
#pragma unroll
                for (int k = 0; k < KS; ++k) {
                    const uint2 part = from[(i * TN + t) * nthreads + k * group_threads];
                    v += ((uint64_t)part.y << 32) | part.x;
                }
                fin[i][t] = v;
            }
    } else {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int t = 0; t < TE; ++t) fin[i][t] = acc[i][t];
    }
    const int ch0 = tn * TN + group * TE;                      // first of this thread's finished channels
    const uint2 *const es0 = reinterpret_cast<uint2 *>(smem + p.e_off) + gtid * strip_e_pitch(TM, TN) + group * TE;
    auto second = [&](int i, int t) -> uint64_t {
        const uint2 e = es0[i * TN + t];
        uint64_t v = ((uint64_t)e.y << 32) | e.x;
#pragma unroll
        for (int k = 1; k < KS; ++k) {
            const uint2 f = es0[k * group_threads * strip_e_pitch(TM, TN) + i * TN + t];
            v += ((uint64_t)f.y << 32) | f.x;
        }
        return v;
    };
    // ---- words above the N low slots: to the next lane by shuffle, across warps through shared memory
    uint2 *xch = xch0 + ((warp << tnx_log2) + tn) * (TM * TE);
    const int lanes_m = 32 >> tnx_log2, lm = lane >> tnx_log2;
    if (UP && lm == lanes_m - 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int t = 0; t < TE; ++t)
                xch[i * TE + t] = make_uint2((uint32_t)(fin[i][t] >> p.SN), HASE ? (uint32_t)(second(i, t) >> p.SN) : 0u);
    }
    __syncthreads();
    const uint2 *xch_in = xch - p.TNX * (TM * TE);
    const bool from_smem = lm == 0 && gtid >= 32;
    const uint32_t keep = xb == 0 ? 0u : 0xFFFFFFFFu;          // nothing comes in at the left end of a row

    const int x = seg * p.XO + xb - p.halo, w0 = x * N - p.col_off;   // group and its first output column
    const int h0 = s_img * TM;
    const int n_rows = min(TM, p.Ho - h0);
    bool col_ok[N];
    int32_t base[N];                                           // what is taken off every sum of slot m
#pragma unroll
    for (int m = 0; m < N; ++m) {
        col_ok[m] = pos_ok && xb >= p.halo && x < p.X && w0 + m >= 0 && w0 + m < p.Wo;
        base[m] = -(KS * moves + 1) * (p.slot_bias[m] + (keep ? p.slot_bias[m + N] : 0));
    }
    const int n_ch = min(TE, p.Co - co0 - ch0);
    const uint32_t mask = p.slot_mask;

    // value[m] of accumulator (i, t)
    auto split = [&](int i, int t, const int32_t (&off)[N], int32_t (&y)[N]) {
        uint64_t q = fin[i][t];
        uint32_t q_in = 0, e_in = 0, qf[N], ef[N];
        uint64_t e = 0;
        if constexpr (HASE) e = second(i, t);
        if constexpr (UP) {
            q_in = __shfl_up_sync(0xFFFFFFFFu, (uint32_t)(q >> p.SN), p.TNX);
            if constexpr (HASE) e_in = __shfl_up_sync(0xFFFFFFFFu, (uint32_t)(e >> p.SN), p.TNX);
            if (from_smem) {
                const uint2 v = xch_in[i * TE + t];
                q_in = v.x;
                if constexpr (HASE) e_in = v.y;
            }
            q_in &= keep;
            if constexpr (HASE) e_in &= keep;
        }
        if constexpr (PACKED_ADD && UP) {                   // the words coming in fill at most the low half, and no slot overflows
            q = (q & 0xFFFFFFFF00000000ull) | (uint32_t)((uint32_t)q + q_in);
            if constexpr (HASE) e = (e & 0xFFFFFFFF00000000ull) | (uint32_t)((uint32_t)e + e_in);
        }
#pragma unroll
        for (int m = 0; m < N; ++m) {
            qf[m] = (m == 0 ? (uint32_t)q : (uint32_t)(q >> (p.S * m))) & mask;
            y[m] = off[m] + (int32_t)qf[m];
            if constexpr (HASE) {
                ef[m] = (m == 0 ? (uint32_t)e : (uint32_t)(e >> (p.S * m))) & mask;
                y[m] += (int32_t)(ef[m] << p.h);
            }
            if constexpr (!PACKED_ADD && UP) {
                if (m < p.up_slots) {
                    y[m] += (int32_t)((q_in >> (p.S * m)) & mask);
                    if constexpr (HASE) y[m] += (int32_t)(((e_in >> (p.S * m)) & mask) << p.h);
                }
            }
        }
    };
    // base plus, on shifted codes, x_off times the channel's weights at the taps that lie inside the image at column w0 + m
    auto offsets = [&](int t, int32_t (&off)[N]) {
#pragma unroll
        for (int m = 0; m < N; ++m) off[m] = base[m];
        if (p.corr && t < n_ch) {
            const int32_t *c = p.corr + co0 + ch0 + t;
#pragma unroll
            for (int m = 0; m < N; ++m)
                if (col_ok[m]) {
                    const int k_lo = max(0, p.pad - w0 - m), k_hi = min(K, p.W + p.pad - w0 - m);
                    off[m] += load_ordered(c + (k_hi - 1) * p.CoP) - (k_lo > 0 ? load_ordered(c + (k_lo - 1) * p.CoP) : 0);   // k_hi >= K - pad > 0
                }
        }
    };
    const int q_shift = p.shift, q_lo = p.lo, q_hi = p.hi;
    auto requant = [&](int32_t v) { return max(q_lo, min(q_hi, v >> q_shift)); };

    if (!p.stage_out) {
        // direct stores; warps whose rows and channels all exist (nearly all) test only the columns
        const size_t chan = (size_t)p.Ho * p.Wo;
        const size_t at = (((size_t)(b0 + db) * p.Co + co0 + ch0) * p.Ho + h0) * p.Wo + w0;
        auto finish = [&](auto *dst, auto full_tag) {
            constexpr bool FULL = decltype(full_tag)::value, REQ = sizeof(*dst) == 1;
            auto *chan_row = dst + at;
#pragma unroll
            for (int t = 0; t < TE; ++t, chan_row += chan) {
                int32_t off[N], y[N];
                offsets(t, off);
                auto *row = chan_row;
#pragma unroll
                for (int i = 0; i < TM; ++i, row += p.Wo) {
                    split(i, t, off, y);
                    if (FULL || (t < n_ch && i < n_rows)) {
#pragma unroll
                        for (int m = 0; m < N; ++m) {
                            if constexpr (REQ) y[m] = requant(y[m]);
                            if (col_ok[m]) row[m] = (std::remove_reference_t<decltype(*dst)>)y[m];
                        }
                    }
                }
            }
        };
        const bool full = __all_sync(0xFFFFFFFFu, n_ch >= TE && (n_rows >= TM || !pos_ok));
        if (p.requant) {
            if (full) finish((int8_t *)p.out, std::true_type());
            else finish((int8_t *)p.out, std::false_type());
        } else {
            if (full) finish((int32_t *)p.out, std::true_type());
            else finish((int32_t *)p.out, std::false_type());
        }
        return;
    }

    // ---- requantised codes staged as bytes [channel][row][column]; with a pool the two rows of a pair are reduced first (the
    // shift and the clamp keep the order, so the maximum is taken before them; only a clamp range that reaches from below 0 to
    // above 127 does not, because the codes above 127 are negative bytes: pool == 2, the maximum of the bytes)
    int8_t *tile = reinterpret_cast<int8_t *>(smem + p.tile_off);
    const int rps = p.pool ? TM / 2 : TM;                      // tile rows per strip
    const int tile_chan = p.TS * rps * p.WTP;
    const int col0 = seg * p.XO * N;                           // first output column of the segment (segments: col_off == 0)
    int8_t *tile_at = tile + ch0 * tile_chan + sl * rps * p.WTP + w0 - col0;
    auto stage_codes = [&](auto pool_tag) {
        constexpr int POOL = decltype(pool_tag)::value;
#pragma unroll
        for (int t = 0; t < TE; ++t) {
            int32_t off[N], y[N], y2[N];
            offsets(t, off);
#pragma unroll
            for (int i = 0; i < TM; i += POOL ? 2 : 1) {
                split(i, t, off, y);
                if constexpr (POOL) {
                    split(i + 1, t, off, y2);
#pragma unroll
                    for (int m = 0; m < N; ++m)
                        y[m] = POOL == 2 ? max((int32_t)(int8_t)requant(y[m]), (int32_t)(int8_t)requant(y2[m])) : max(y[m], y2[m]);
                }
#pragma unroll
                for (int m = 0; m < N; ++m)
                    if (col_ok[m]) tile_at[t * tile_chan + (POOL ? i / 2 : i) * p.WTP + m] = (int8_t)(POOL == 2 ? y[m] : requant(y[m]));
            }
        }
    };
    if (p.pool == 1) stage_codes(std::integral_constant<int, 1>());
    else if (p.pool) stage_codes(std::integral_constant<int, 2>());
    else stage_codes(std::integral_constant<int, 0>());
    __syncthreads();

    // ---- staged codes leave the CTA in pieces of `vec` bytes along a row, neighbouring columns reduced first with a pool
    const int sh = p.pool ? 1 : 0, rps_log2 = 31 - __clz(rps);
    const int Hq = p.Ho >> sh, Wq = p.Wo >> sh;
    const int wn = (p.NSEG > 1 ? min(p.Wo - col0, p.XO * N) : p.Wo) >> sh;   // output columns of this segment
    const int ncv = min(p.TCO, p.Co - co0), tr = TSe * rps;
    const int ppr = p.out_bits < 8 ? ((wn * p.out_bits) >> 3) / p.vec : wn / p.vec;
    const float inv_ppr = 1.0f / (float)ppr, inv_tr = 1.0f / (float)tr;
    for (int idx = tid; idx < ncv * tr * ppr; idx += nthreads) {
        const int rr = small_div(idx, ppr, inv_ppr), piece = idx - rr * ppr;
        const int cl = small_div(rr, tr, inv_tr), r = rr - cl * tr;
        const int ts = s0 + (r >> rps_log2), d = fast_div(ts, p.mg_sh);
        const int hq = (ts - d * p.SH) * rps + (r & (rps - 1));
        if (hq >= Hq) continue;                                // rows past the image in its last strip
        const int8_t *src = tile + cl * tile_chan + r * p.WTP;
        const size_t e0 = (((size_t)(b0 + d) * p.Co + co0 + cl) * Hq + hq) * Wq + (col0 >> sh);   // first code of this segment's row
        if (p.out_bits < 8) {
            // dense codes: every output byte gathers 8 / out_bits neighbouring codes (rows and segments start on byte
            // boundaries, checked on the host)
            const int ob = p.out_bits, cpb = 8 / ob;
            const uint32_t cmask = (1u << ob) - 1u;
            uint8_t *dst = (uint8_t *)p.out + ((e0 * ob) >> 3) + piece * p.vec;
            uint32_t word = 0;
            for (int u = 0; u < p.vec * cpb; ++u) {
                const int col = piece * p.vec * cpb + u;
                int v = src[p.pool ? 2 * col : col];
                if (p.pool) {
                    int v1 = src[2 * col + 1];
                    if (!p.out_signed) { v &= 0xFF; v1 &= 0xFF; }
                    v = max(v, v1);
                }
                word |= ((uint32_t)v & cmask) << (ob * u);
            }
            if (p.vec == 4) *reinterpret_cast<uint32_t *>(dst) = word;
            else *dst = (uint8_t)word;
        } else {                                               // one code per byte: staged only for a pool
            int8_t *dst = (int8_t *)p.out + e0 + piece * p.vec;
            src += 2 * piece * p.vec;
            if (p.vec == 8) {
                const uint4 v = *reinterpret_cast<const uint4 *>(src);
                *reinterpret_cast<uint2 *>(dst) = p.out_signed ? make_uint2(pool_pairs<true>(v.x, v.y, v.x, v.y), pool_pairs<true>(v.z, v.w, v.z, v.w))
                                                               : make_uint2(pool_pairs<false>(v.x, v.y, v.x, v.y), pool_pairs<false>(v.z, v.w, v.z, v.w));
            } else if (p.vec == 4) {
                const uint2 v = *reinterpret_cast<const uint2 *>(src);
                *reinterpret_cast<uint32_t *>(dst) = p.out_signed ? pool_pairs<true>(v.x, v.y, v.x, v.y) : pool_pairs<false>(v.x, v.y, v.x, v.y);
            } else {
                int a = src[0], b = src[1];
                if (!p.out_signed) { a &= 0xFF; b &= 0xFF; }
                *dst = (int8_t)max(a, b);
            }
        }
    }
}

template <int N, int KT, int JT, int TM, int TN, int KS = 1>
static int launch_strip_tile(const StripLaunch &s, cudaStream_t st) {
    auto run = [&](auto kern) -> int {
        return with_dynamic_smem(reinterpret_cast<const void *>(kern), s.smem_bytes,
                                 [&] { return launch_dependent(kern, s.grid, dim3(s.threads), s.smem_bytes, st, s.p); });
    };
    if (s.moves) return s.sp ? run(conv2d_strip_kernel<N, KT, JT, TM, TN, true, true, KS>) : run(conv2d_strip_kernel<N, KT, JT, TM, TN, false, true, KS>);
    return s.sp ? run(conv2d_strip_kernel<N, KT, JT, TM, TN, true, false, KS>) : run(conv2d_strip_kernel<N, KT, JT, TM, TN, false, false, KS>);
}

template <int N, int KT, int JT>
int strip_wait_timeouts(unsigned int *h_count) {
    return cudaMemcpyFromSymbol(h_count, strip_timeouts, sizeof(*h_count)) == cudaSuccess ? HIKONV_OK : HIKONV_ERR_CUDA;
}

template <int N, int KT, int JT>
int launch_strip(const StripLaunch &s, cudaStream_t st) {
    if constexpr (KT > 0) {
        if (s.TM == 2 && s.TN == 4 && s.KS == 2) return launch_strip_tile<N, KT, JT, 2, 4, 2>(s, st);
        if (s.TM == 2 && s.TN == 8 && s.KS == 2) return launch_strip_tile<N, KT, JT, 2, 8, 2>(s, st);
        if (s.TM == 2 && s.TN == 4 && s.KS == 4) return launch_strip_tile<N, KT, JT, 2, 4, 4>(s, st);
    }
    if (s.KS != 1) return HIKONV_ERR_UNSUPPORTED;
    if (s.TM == 2 && s.TN == 4) return launch_strip_tile<N, KT, JT, 2, 4>(s, st);
    if (s.TM == 2 && s.TN == 8) return launch_strip_tile<N, KT, JT, 2, 8>(s, st);
    if (s.TM == 4 && s.TN == 8) return launch_strip_tile<N, KT, JT, 4, 8>(s, st);
    return HIKONV_ERR_UNSUPPORTED;
}

}  // namespace hikonv
