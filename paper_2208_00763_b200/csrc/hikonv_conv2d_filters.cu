// The packed method with one activation and the weights of several filters in a multiplication, for 3x3 layers of few input channels.
//
// A word holds the weights of three filters at one tap, S = 17 bits apart (Eq. 5 on the filters):  B = sum_s w[co + s][tap] 2^(S s).
// Its product with ONE activation has the products of all three filters in its slots, and slots never overlap, so the sums over input
// channels, kernel rows and kernel columns all stay packed: no carry reaches a neighbouring pixel, and slots as wide as the
// layer's sums need no moves.  The multiplier is the 53-bit one of the double-precision unit.  Every value it sees is an integer:
// products are exact, and the accumulator, which starts at 2^52 plus a bias that keeps every slot non-negative, stays in
// [2^52, 2^53), where doubles are the integers; its fraction bits are the slots.
//
// Where codes are wide the words of pixels and taps (hikonv_conv2d_strip.cuh) hold three products, too, at 4.8 cycles a warp-wide
// multiplication in their loop; a double-precision one takes 2.02 (hikonv_pipe_rate), and other instructions issue beside it.  The first layer of the
// compact CNN spent three quarters of its instructions outside the multiplications (prologue, exchange of upper slots, split,
// staging of bytes); here the split needs no neighbour and the 2x2 pool is a thread's own pixels.
//
// A thread owns 2 x 2 output pixels (a pooling window) and NW words; lanes run along the pixels, so the words are the same for
// a warp.  CTAs stay: each packs the weights of its filters once and walks over tiles; while it multiplies one step (a tile's
// activations as doubles in shared memory) its threads fetch the next one's, a few rows of four codes beside every channel, into the
// other buffer.  A layer is one launch and writes no packed activations.
// First layer of the network (64x3x160x320 -> 16 channels, u8 x s4, pooled), packing launch included, as a graph: 122.9 -> 82 us (97.5 with one
// tile a CTA, staged before it multiplies).  What bounds it: instructions around the multiplies.  Of 54.3 M warp instructions 17.0 M are
// double-precision; the schedulers issue in 59 % of the cycles, the pipe is busy in 37 %, and warps wait for results of their own
// and for their turn, hardly for the barrier or for loads.
#include "hikonv_cuda.cuh"
#include "hikonv_conv2d_filters.h"
#include "hikonv_conv2d_util.cuh"

namespace hikonv {

constexpr int kRows = 2;                 // rows of four codes that a thread fetches for the next step beside one channel's products
constexpr int kWords = 4;                // kernel words of a thread whose codes are loaded together

// 2^52 + byte b of v.
__device__ __forceinline__ double byte_as_double(uint32_t v, int b) { return __hiloint2double(0x43300000, (int)extract_code<false>(v, b)); }

// The aligned words that hold the four codes from column col0 on of an image row of W one-byte codes, which starts at code `row` of the
// tensor x: the codes begin at byte `off` of lo and go on in hi.  Words without a code of the row are not read and left alone, and hi
// is not needed where off is zero.  RAGGED: the tensor's ends need not be aligned, and the words that reach outside it are put
// together from bytes (`codes`: all of the tensor).
template <bool RAGGED>
__device__ __forceinline__ void load_row_codes(const int8_t *x, int row, int codes, int W, int col0, uint32_t &lo, uint32_t &hi, uint32_t &off) {
    const int8_t *src = x + (row + col0);
    off = (uint32_t)(uintptr_t)src & 3u;
    const uint32_t *al = reinterpret_cast<const uint32_t *>(src - off);
    const int c = col0 - (int)off;                               // column at the start of lo
    auto load = [&](int i, uint32_t &v) {
        const int first = row + c + 4 * i;                       // code at the start of the word
        if (!RAGGED || (first >= 0 && first <= codes - 4)) v = load_ordered(al + i);
        else
            for (int b = 0; b < 4; ++b)
                if (c + 4 * i + b >= 0 && c + 4 * i + b < W) v |= (uint32_t)(uint8_t)load_ordered(x + first + b) << (8 * b);
    };
    if (c + 3 >= 0 && c < W) load(0, lo);
    if (off != 0u && c + 7 >= 0 && c + 4 < W) load(1, hi);
}

// RAGGED: the input begins at any byte, or ends at any (an instantiation of its own: the branch for it cost aligned inputs 2 %).
template <int NW, bool RAGGED>
__global__ void __launch_bounds__(kFiltersThreads, filters_resident(NW)) conv2d_filters_kernel(const __grid_constant__ FiltersParams p) {
    constexpr int NS = kFiltersSlots, S = kFiltersSlotBits, KT = kFiltersK, KK = KT * KT, AC = KT + 1;   // AC: columns of a row that a thread's pixels read
    extern __shared__ __align__(16) double smem_d[];
    grid_dependency_release();

    const int tid = threadIdx.x, nthreads = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int word0 = blockIdx.y * p.WT;
    // warps: positions fastest, then groups of words
    int wp = warp, group = 0;
    while (wp >= p.pos_warps) { wp -= p.pos_warps; ++group; }
    const int pos = wp * 32 + lane, sl = fast_div(pos, p.mg_tq), xq = pos - sl * p.TQ;

    // shared memory: kernel words [channel, tap][word], two buffers of activations [channel][row][column]
    double *const Bs = smem_d, *const As = smem_d + (size_t)p.Ci * KK * p.WT;
    const int a_words = p.CK * p.plane;

    // Staging: a thread keeps its four columns of a step's rows and walks down the rows of all its channels.
    const int hw = p.H * p.W, pw4 = p.PW >> 2, a_step = nthreads / pw4;
    const int a_lane = tid / pw4, a_col = tid - a_lane * pw4, a_first = a_lane < a_step ? a_lane : 0x3FFFFFFF;
    const int a_first_c = a_lane / p.rows, a_first_r = a_lane - a_first_c * p.rows;
    const int a_step_c = a_step / p.rows, a_step_r = a_step - a_step_c * p.rows;
    const uint32_t code_flip = p.x_signed ? 0x80808080u : 0u;  // signed bytes as unsigned ones, 128 too large
    const double code_zero = 4503599627370496.0 + (p.x_signed ? 128.0 : 0.0);
    // the step that is fetched: its tile, first channel and buffer, and the thread's next row of it
    int n_tile = blockIdx.x, n_ci0 = 0, n_rows = 0, n_row = 0, n_c = 0, n_r = 0, n_b0 = 0, n_h0 = 0, n_col0 = 0;
    double *n_buf = As;
    auto begin_fetch = [&]() {
        const int strip_tile = n_tile / p.NSEG, seg = n_tile - strip_tile * p.NSEG, g0 = strip_tile * p.TS;
        n_b0 = g0 / p.SH;
        n_h0 = 2 * (g0 - n_b0 * p.SH);
        n_col0 = seg * 2 * p.TQ - p.pad + 4 * a_col;
        n_rows = n_tile < p.tiles ? min(p.CK, p.Ci - n_ci0) * p.rows : 0;
        n_row = a_first;
        n_c = a_first_c;
        n_r = a_first_r;
    };
    uint32_t f_lo[kRows], f_hi[kRows], f_off[kRows];
    int f_at[kRows];                                           // where a row's doubles go (-1: nowhere)
    auto fetch_rows = [&]() {
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            f_lo[u] = f_hi[u] = f_off[u] = 0u;
            f_at[u] = -1;
            if (n_row >= n_rows) continue;
            f_at[u] = n_c * p.plane + n_r * p.PW + 4 * a_col;
            const int d = fast_div(n_h0 + n_r, p.mg_hp), b = n_b0 + d, h = n_h0 + n_r - d * p.Hp - p.pad;
            if (b < p.B && h >= 0 && h < p.H)
                load_row_codes<RAGGED>(p.x, (b * p.Ci + n_ci0 + n_c) * hw + h * p.W, p.codes, p.W, n_col0, f_lo[u], f_hi[u], f_off[u]);   // (fewer than 2^31 codes)
            n_row += a_step;
            n_c += a_step_c;
            n_r += a_step_r;
            if (n_r >= p.rows) { n_r -= p.rows; ++n_c; }
        }
    };
    auto put_rows = [&]() {
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            if (f_at[u] < 0) continue;
            const uint32_t v = (__funnelshift_r(f_lo[u], f_hi[u], 8 * f_off[u]) & byte_range_mask(0, -n_col0, p.W - n_col0)) ^ code_flip;
            double2 *dst = reinterpret_cast<double2 *>(n_buf + f_at[u]);
            dst[0] = make_double2(byte_as_double(v, 0) - code_zero, byte_as_double(v, 1) - code_zero);
            dst[1] = make_double2(byte_as_double(v, 2) - code_zero, byte_as_double(v, 3) - code_zero);
        }
    };

    double acc[2][2][NW];
    const double start = 4503599627370496.0 + p.bias;
    auto clear = [&]() {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int w = 0; w < NW; ++w) acc[i][j][w] = start;
    };

    // ---- split and store the thread's pixels of a tile
    auto finish_tile = [&](int b_img, int s_img, int seg, bool pos_ok) {
        const int h0 = 2 * s_img, col = seg * 2 * p.TQ + 2 * xq;
        const bool live = pos_ok && col < p.Wo, two_cols = col + 1 < p.Wo, two_rows = h0 + 1 < p.Ho;
        auto requant = [&](int32_t v) { return max(p.lo, min(p.hi, v >> p.shift)); };
        const size_t plane_out = p.pool ? (size_t)(p.Ho >> 1) * (p.Wo >> 1) : (size_t)p.Ho * p.Wo;
        const size_t at_out = ((size_t)b_img * p.Co + word0 * NS) * plane_out +
                              (p.pool ? (size_t)s_img * (p.Wo >> 1) + (col >> 1) : (size_t)h0 * p.Wo + col);
        // word wl of the CTA, f: the fraction bits of its four pixels
        auto finish = [&](int wl, const uint64_t (&f)[2][2]) {
            const int left = p.Co - (word0 + wl) * NS;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                if (s >= left) break;
                int32_t y[2][2];                                   // the fields, still with their bias
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        uint32_t v = (uint32_t)(f[i][j] >> (S * s));
                        if (s < NS - 1) v &= (1u << S) - 1u;
                        y[i][j] = (int32_t)v;
                    }
                const size_t at = at_out + (size_t)(wl * NS + s) * plane_out;
                if (p.pool) {
                    // the shift and the clamp keep the order, but for codes from below 0 to above 127 the bytes do not (pool == 2)
                    int32_t m = max(max(y[0][0], y[0][1]), max(y[1][0], y[1][1]));
                    if (p.pool == 2) {
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int j = 0; j < 2; ++j) y[i][j] = (int32_t)(int8_t)requant(y[i][j] - p.slot_bias);
                        m = max(max(y[0][0], y[0][1]), max(y[1][0], y[1][1]));
                    } else m = requant(m - p.slot_bias);
                    ((int8_t *)p.out)[at] = (int8_t)m;
                    continue;
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (i == 1 && !two_rows) continue;
                    const int32_t y0 = y[i][0] - p.slot_bias, y1 = y[i][1] - p.slot_bias;
                    if (p.requant) {
                        int8_t *dst = (int8_t *)p.out + at + i * p.Wo;
                        const int32_t v0 = requant(y0), v1 = requant(y1);
                        if (p.pair_stores) *reinterpret_cast<uint16_t *>(dst) = (uint16_t)((v0 & 0xFF) | (v1 << 8));
                        else {
                            dst[0] = (int8_t)v0;
                            if (two_cols) dst[1] = (int8_t)v1;
                        }
                    } else {
                        int32_t *dst = (int32_t *)p.out + at + i * p.Wo;
                        if (p.pair_stores) *reinterpret_cast<int2 *>(dst) = make_int2(y0, y1);
                        else {
                            dst[0] = y0;
                            if (two_cols) dst[1] = y1;
                        }
                    }
                }
            }
        };
        constexpr uint64_t kFraction = (1ull << 52) - 1;
        if (!live) return;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            uint64_t f[2][2];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) f[i][j] = (uint64_t)__double_as_longlong(acc[i][j][w]) & kFraction;
            finish(group * NW + w, f);
        }
    };

    grid_dependency_wait();                                    // the input may come from the kernel before
    begin_fetch();
    while (n_row < n_rows) {
        fetch_rows();
        put_rows();
    }
    // kernel words of all input channels
    {
        const int n = p.Ci * KK, items = p.WT * n;
        const float inv_n = 1.0f / (float)n;
        for (int it0 = tid; it0 < items; it0 += kWords * nthreads) {
            int32_t v[kWords][NS];
            int at[kWords];
#pragma unroll
            for (int u = 0; u < kWords; ++u) {
                const int it = min(it0 + u * nthreads, items - 1);     // (threads past the last word repeat it)
                const int wl = small_div(it, n, inv_n), e = it - wl * n, co = (word0 + wl) * NS;
                const int8_t *src = p.w + (size_t)co * n + e;
                at[u] = e * p.WT + wl;
#pragma unroll
                for (int s = 0; s < NS; ++s) v[u][s] = co + s < p.Co ? (int32_t)load_ordered(src + (size_t)s * n) : 0;
            }
#pragma unroll
            for (int u = 0; u < kWords; ++u) {
                double b = 0.0;
#pragma unroll
                for (int s = NS - 1; s >= 0; --s) b = fma(b, (double)(1 << S), (double)(p.w_signed ? v[u][s] : v[u][s] & 0xFF));
                Bs[at[u]] = b;
            }
        }
    }
    __syncthreads();

    int buf = 0;
    clear();
    for (int tile = blockIdx.x, ci0 = 0; tile < p.tiles;) {
        // ---- one step: the products of up to CK input channels of a tile, and beside them the fetch of the next step's activations
        const int ckn = min(p.CK, p.Ci - ci0);
        const bool last = ci0 + p.CK >= p.Ci;
        n_tile = last ? tile + (int)gridDim.x : tile;
        n_ci0 = last ? 0 : ci0 + p.CK;
        n_buf = As + (buf ^ 1) * a_words;
        begin_fetch();
        const int strip_tile = tile / p.NSEG, seg = tile - strip_tile * p.NSEG, g0 = strip_tile * p.TS;
        const int b0 = g0 / p.SH, s0 = g0 - b0 * p.SH;
        const bool pos_ok = sl < p.TS && g0 + sl < p.strips;
        const int db = fast_div(s0 + (pos_ok ? sl : 0), p.mg_sh), s_img = s0 + (pos_ok ? sl : 0) - db * p.SH;
        const double *a_c = As + buf * a_words + (db * p.Hp + (s_img - s0) * 2) * p.PW + 2 * xq;
        const double *b_c = Bs + ci0 * (KK * p.WT) + group * NW;
        for (int c = 0; c < ckn; ++c, a_c += p.plane, b_c += KK * p.WT) {
            fetch_rows();
            double a[KT + 1][AC];
#pragma unroll
            for (int r = 0; r <= KT; ++r)
#pragma unroll
                for (int k = 0; k < AC; k += 2) {
                    const double2 v = *reinterpret_cast<const double2 *>(a_c + r * p.PW + k);
                    a[r][k] = v.x;
                    a[r][k + 1] = v.y;
                }
#pragma unroll
            for (int kh = 0; kh < KT; ++kh)
#pragma unroll
                for (int kw = 0; kw < KT; ++kw) {
                    double b[NW];
#pragma unroll
                    for (int w = 0; w < NW; w += 2) {
                        const double2 v = *reinterpret_cast<const double2 *>(b_c + (kh * KT + kw) * p.WT + w);
                        b[w] = v.x;
                        b[w + 1] = v.y;
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
#pragma unroll
                            for (int w = 0; w < NW; ++w) acc[i][j][w] = fma(a[kh + i][kw + j], b[w], acc[i][j][w]);
                }
            put_rows();
        }
        while (n_row < n_rows) {
            fetch_rows();
            put_rows();
        }
        if (last) {
            finish_tile(b0 + db, s_img, seg, pos_ok);
            clear();
        }
        __syncthreads();
        buf ^= 1;
        tile = n_tile;
        ci0 = n_ci0;
    }
}

template <int NW>
static int launch_filters_as(const FiltersLaunch &l, cudaStream_t st) {
    auto launch = [&](auto kern) {
        return with_dynamic_smem(reinterpret_cast<const void *>(kern), l.smem_bytes,
                                 [&] { return launch_dependent(kern, l.grid, dim3(l.threads), l.smem_bytes, st, l.p); });
    };
    return (((uintptr_t)l.p.x | (unsigned)l.p.codes) & 3) != 0 ? launch(conv2d_filters_kernel<NW, true>) : launch(conv2d_filters_kernel<NW, false>);
}

int launch_filters(const FiltersLaunch &l, cudaStream_t st) {
    switch (l.NW) {
        case 2: return launch_filters_as<2>(l, st);
        case 4: return launch_filters_as<4>(l, st);
        case 6: return launch_filters_as<6>(l, st);
        default: return HIKONV_ERR_UNSUPPORTED;
    }
}

}  // namespace hikonv
