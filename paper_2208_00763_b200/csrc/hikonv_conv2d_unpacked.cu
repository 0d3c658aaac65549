// The comparator of hikonv_conv2d (HIKONV_ALGO_UNPACKED_IMAD): one product per 32-bit multiply-add, int32 accumulators, codes
// and weights staged as 32-bit words.  A CTA computes TR consecutive output rows (one row segment each) times TCO output
// channels; each thread owns eight positions (dealt round-robin to the lanes of a warp) times four channels.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "hikonv_cuda.cuh"
#include "hikonv_conv2d_output.h"
#include "hikonv_conv2d_unpacked.h"
#include "hikonv_conv2d_util.cuh"

namespace hikonv {

constexpr int kUThreads = 256;
constexpr int kUPieces = 4;              // 16-byte pieces per thread and stage whose offsets are kept in registers
constexpr int kUTM = 8, kUTN = 4;        // per-thread tile

// KT: kernel size when known at compile time (0: read from the parameters); PITCH: words per row in shared memory likewise.
template <int KT, int PITCH>
__global__ void __launch_bounds__(kUThreads, 2) conv2d_unpacked_kernel(const UnpackedParams p) {
    constexpr int TM = kUTM, TN = kUTN;
    extern __shared__ __align__(16) uint32_t smem[];
    grid_dependency_release();
    uint32_t *As = smem;                                   // two tiles [CK][a_plane]
    uint32_t *Bs = smem + p.b_off;                         // two tiles [CK*K*K][TCO]

    const int tid = threadIdx.x, nthreads = blockDim.x;
    const int tnx_log2 = 31 - __clz(p.TNX);                 // TNX is a power of two
    const int tn = tid & (p.TNX - 1);
    const int row_tile = p.NSEG > 1 ? (int)(blockIdx.x / (unsigned)p.NSEG) : (int)blockIdx.x;
    const int seg = blockIdx.x - row_tile * p.NSEG;
    const int R0 = row_tile * p.TR;
    const int co0 = blockIdx.y * p.TCO;
    const int TRe = min(p.TR, p.total_rows - R0);
    const int b0 = R0 / p.Ho, h0 = R0 - b0 * p.Ho;
    const int Rp0 = b0 * p.Hp + h0;                         // first staged padded row
    const int Rlast = R0 + TRe - 1;
    const int bl = b0 + fast_div(h0 + TRe - 1, p.mg_ho);
    const int NR = (bl * p.Hp + (Rlast - bl * p.Ho) + p.K - 1) - Rp0 + 1;
    const int TP = TRe * p.XB;                              // positions of this tile

    const int lane = tid & 31, warp = tid >> 5;
    const int lanes_m = 32 >> tnx_log2, lm = lane >> tnx_log2;
    const int wpos0 = warp * lanes_m * TM;
    const uint32_t *aptr[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        // an idle position (past the tile) reads the words of position 0; its result is dropped
        const int pos = wpos0 + i * lanes_m + lm, pc = pos < TP ? pos : 0;
        const int r = fast_div(pc, p.mg_xb), xb = pc - r * p.XB;
        const int db = fast_div(h0 + r, p.mg_ho);           // images past the tile's first one: K - 1 more padded rows each
        aptr[i] = As + p.lead + (r + db * (p.K - 1)) * p.XBS + xb;
    }
    int32_t acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int t = 0; t < TN; ++t) acc[i][t] = 0;

    const int KJ = p.K * p.K;
    const int xq = (p.XB + 3) / 4;                                   // 16-byte pieces per row
    const int ap_plane = p.B * p.Hp * p.XBT;
    const uint32_t *ap_tile = p.ap + (size_t)Rp0 * p.XBT + seg * p.XO;

    // the pieces of a stage this thread copies: the same ones every stage (channel in the top byte of the destination, -1: none)
    int piece_src[kUPieces], piece_dst[kUPieces];
#pragma unroll
    for (int k = 0; k < kUPieces; ++k) {
        const int q = tid + k * nthreads;                            // numbered [row][channel][piece of the row]
        const int rc = fast_div(q, p.mg_xq), qd = q - rc * xq;
        const int rl = fast_div(rc, p.mg_ck), cl = rc - rl * p.CK;
        piece_src[k] = cl * ap_plane + rl * p.XBT + 4 * qd;
        piece_dst[k] = q < p.CK * NR * xq ? ((cl << 24) | (cl * p.a_plane + p.lead + rl * p.XBS + 4 * qd)) : -1;
    }
    const bool pieces_in_regs = p.CK * NR * xq <= kUPieces * nthreads;
    const int tco4 = p.TCO / 4, tco4_log2 = 31 - __clz(tco4);        // TCO / 4 is a power of two

    auto fetch = [&](int ci0, int ckn, uint32_t *Adst, uint32_t *Bdst) {
        const uint32_t *asrc = ap_tile + (size_t)ci0 * ap_plane;
        if (pieces_in_regs) {
#pragma unroll
            for (int k = 0; k < kUPieces; ++k)
                if (piece_dst[k] >= 0 && (piece_dst[k] >> 24) < ckn) cp_async_16(Adst + (piece_dst[k] & 0xFFFFFF), asrc + piece_src[k]);
        } else {
            const int per_ch = NR * xq;
            for (int cl = 0; cl < ckn; ++cl) {
                const uint32_t *src = asrc + (size_t)cl * ap_plane;
                uint32_t *dst = Adst + cl * p.a_plane + p.lead;
                for (int idx = tid; idx < per_ch; idx += nthreads) {
                    const int rl = fast_div(idx, p.mg_xq), qd = idx - rl * xq;
                    cp_async_16(dst + rl * p.XBS + 4 * qd, src + (size_t)rl * p.XBT + 4 * qd);
                }
            }
        }
        const uint32_t *bsrc = p.wp + (size_t)ci0 * KJ * p.CoP + co0;
        const int rows_b = ckn * KJ;
        for (int idx = tid; idx < rows_b << tco4_log2; idx += nthreads) {
            const int kr = idx >> tco4_log2, c4 = idx & (tco4 - 1);
            uint32_t *dst = Bdst + kr * kBPitch + c4 * 4;
            if (co0 + c4 * 4 < p.CoP) cp_async_16(dst, bsrc + kr * p.CoP + c4 * 4);
            else *reinterpret_cast<uint4 *>(dst) = make_uint4(0, 0, 0, 0);
        }
        cp_async_commit();
    };

    grid_dependency_wait();                                          // everything above touched no global memory
    fetch(0, min(p.CK, p.Ci), As, Bs);
    int stage = 0;
    for (int ci0 = 0; ci0 < p.Ci; ci0 += p.CK, stage ^= 1) {
        const int ckn = min(p.CK, p.Ci - ci0);
        cp_async_wait_all();
        __syncthreads();                                             // this stage has landed; the previous one is fully consumed
        if (ci0 + p.CK < p.Ci)
            fetch(ci0 + p.CK, min(p.CK, p.Ci - ci0 - p.CK), As + (stage ^ 1) * p.a_words, Bs + (stage ^ 1) * p.b_words);
        const int astage = stage * p.a_words;
        const uint32_t *bptr = Bs + stage * p.b_words + tn * TN;
        if constexpr (KT > 0) {
            const uint32_t *ap[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i) ap[i] = aptr[i] + astage;
            const uint32_t *bp = bptr;
            // two channels per iteration: the operand loads of the next step then rotate through register
            // names instead of being copied at the loop edge
#pragma unroll 2
            for (int cl = 0; cl < ckn; ++cl) {
#pragma unroll
                for (int kh = 0; kh < KT; ++kh) {
#pragma unroll
                    for (int j = 0; j < KT; ++j) {
                        uint32_t a[TM];
#pragma unroll
                        for (int i = 0; i < TM; ++i) a[i] = ap[i][kh * PITCH - j];
                        const uint4 v = *reinterpret_cast<const uint4 *>(bp + (kh * KT + j) * kBPitch);
                        const uint32_t b[TN] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int i = 0; i < TM; ++i)
#pragma unroll
                            for (int t = 0; t < TN; ++t) acc[i][t] += (int32_t)a[i] * (int32_t)b[t];
                    }
                }
#pragma unroll
                for (int i = 0; i < TM; ++i) ap[i] += p.a_plane;
                bp += KT * KT * kBPitch;
            }
        } else {
            for (int cl = 0; cl < ckn; ++cl) {
                for (int kh = 0; kh < p.K; ++kh) {
                    for (int j = 0; j < p.K; ++j) {
                        const int aoff = astage + cl * p.a_plane + kh * p.XBS - j;
                        const uint4 v = *reinterpret_cast<const uint4 *>(bptr + ((cl * p.K + kh) * p.K + j) * kBPitch);
                        const uint32_t b[TN] = {v.x, v.y, v.z, v.w};
                        uint32_t a[TM];
#pragma unroll
                        for (int i = 0; i < TM; ++i) a[i] = aptr[i][aoff];
#pragma unroll
                        for (int i = 0; i < TM; ++i)
#pragma unroll
                            for (int t = 0; t < TN; ++t) acc[i][t] += (int32_t)a[i] * (int32_t)b[t];
                    }
                }
            }
        }
    }

    // where each position's pixel goes: element offset relative to the CTA's first output (image b0, channel co0), which fits
    // 32 bits (checked on the host); -1: none
    uint32_t pix_rel[TM];
    bool pix_ok[TM];
    int tile_pos[TM];                                                // staged output: byte offset of the pixel in a channel's tile
    const uint32_t chan_stride = (uint32_t)(p.Ho * p.Wo);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int pos = wpos0 + i * lanes_m + lm, pc = pos < TP ? pos : 0;
        const int r = fast_div(pc, p.mg_xb), xbl = pc - r * p.XB;
        const int xg = seg * p.XO + xbl - p.K;                       // output column; halo positions give no pixels
        const int db = fast_div(h0 + r, p.mg_ho);
        const int h = h0 + r - db * p.Ho;
        pix_ok[i] = pos < TP && xbl >= p.K && xg < p.X;
        pix_rel[i] = (uint32_t)(db * p.Co) * chan_stride + (uint32_t)(h * p.Wo + xg);
        tile_pos[i] = r * p.WTP + (xbl - p.K);
    }
    const size_t cta_off = ((size_t)b0 * p.Co + co0) * chan_stride;

    if (p.stage_out) __syncthreads();                                // the staged tile reuses the operand buffers of the main loop
    int8_t *tile = reinterpret_cast<int8_t *>(smem);
    const int tile_chan = p.TR * p.WTP;                              // bytes per channel of the staged tile
    auto finish = [&](auto requant_tag, auto staged_tag) {
        constexpr bool REQ = decltype(requant_tag)::value, STAGED = decltype(staged_tag)::value;
        int8_t *out8 = (int8_t *)p.out + cta_off;
        int32_t *out32 = (int32_t *)p.out + cta_off;
#pragma unroll
        for (int t = 0; t < TN; ++t) {
            const int cl = tn * TN + t;
            const uint32_t chan_rel = (uint32_t)cl * chan_stride;
            const bool chan_ok = co0 + cl < p.Co;
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                if (!chan_ok || !pix_ok[i]) continue;
                int32_t v = acc[i][t];
                if constexpr (REQ) {
                    v = max(p.lo, min(p.hi, v >> p.shift));
                    if constexpr (STAGED) tile[cl * tile_chan + tile_pos[i]] = (int8_t)v;
                    else out8[pix_rel[i] + chan_rel] = (int8_t)v;
                } else {
                    out32[pix_rel[i] + chan_rel] = v;
                }
            }
        }
    };
    if (!p.requant) finish(std::false_type(), std::false_type());
    else if (p.stage_out) finish(std::true_type(), std::true_type());
    else finish(std::true_type(), std::false_type());
    if (!p.stage_out) return;

    // staged codes leave the CTA: whole rows in pieces of `vec` bytes, optionally max-pooled 2x2 on the way
    __syncthreads();
    const int col0 = seg * p.XO;                                     // first output column of this row segment
    const int wn = min(p.Wo - col0, p.XO);                           // columns of this segment
    const int ncv = min(p.TCO, p.Co - co0);                          // channels of this tile that exist
    const int sh = p.pool ? 1 : 0;
    const int Hq = p.Ho >> sh, Wq = p.Wo >> sh, TRq = TRe >> sh;
    const int ppr = p.out_bits < 8 ? (((wn >> sh) * p.out_bits) >> 3) / p.vec : (wn >> sh) / p.vec;
    const float inv_ppr = 1.0f / (float)ppr, inv_tr = 1.0f / (float)TRq;
    for (int idx = tid; idx < ncv * TRq * ppr; idx += nthreads) {
        const int rr = small_div(idx, ppr, inv_ppr), piece = idx - rr * ppr;
        const int cl = small_div(rr, TRq, inv_tr), rq = rr - cl * TRq;
        const int r = rq << sh;
        const int db = fast_div(h0 + r, p.mg_ho);
        const int b = b0 + db, h = h0 + r - db * p.Ho;
        const int8_t *src = tile + cl * tile_chan + r * p.WTP;
        const size_t e0 = ((((size_t)b * p.Co + co0 + cl) * Hq + (h >> sh)) * Wq + (col0 >> sh));   // first code of this segment's row
        if (p.out_bits < 8) {
            const int ob = p.out_bits, cpb = 8 / ob;
            const uint32_t cmask = (1u << ob) - 1u;
            uint8_t *dst = (uint8_t *)p.out + ((e0 * ob) >> 3) + piece * p.vec;
            uint32_t word = 0;
            for (int u = 0; u < p.vec * cpb; ++u) {
                const int col = piece * p.vec * cpb + u;             // code index within the segment's (pooled) row
                int v;
                if (p.pool) {
                    int a0 = src[2 * col], a1 = src[2 * col + 1], c0 = src[p.WTP + 2 * col], c1 = src[p.WTP + 2 * col + 1];
                    if (!p.out_signed) { a0 &= 0xFF; a1 &= 0xFF; c0 &= 0xFF; c1 &= 0xFF; }
                    v = max(max(a0, a1), max(c0, c1));
                } else {
                    v = src[col];
                }
                word |= ((uint32_t)v & cmask) << (ob * u);
            }
            if (p.vec == 4) *reinterpret_cast<uint32_t *>(dst) = word;
            else *dst = (uint8_t)word;
        } else {
            src += 2 * piece * p.vec;                                // one code per byte: staged only for a pool
            int8_t *dst = (int8_t *)p.out + e0 + piece * p.vec;
            if (p.vec == 8) {
                const uint4 r0 = *reinterpret_cast<const uint4 *>(src), r1 = *reinterpret_cast<const uint4 *>(src + p.WTP);
                *reinterpret_cast<uint2 *>(dst) = p.out_signed ? make_uint2(pool_pairs<true>(r0.x, r0.y, r1.x, r1.y), pool_pairs<true>(r0.z, r0.w, r1.z, r1.w))
                                                               : make_uint2(pool_pairs<false>(r0.x, r0.y, r1.x, r1.y), pool_pairs<false>(r0.z, r0.w, r1.z, r1.w));
            } else if (p.vec == 4) {
                const uint2 r0 = *reinterpret_cast<const uint2 *>(src), r1 = *reinterpret_cast<const uint2 *>(src + p.WTP);
                *reinterpret_cast<uint32_t *>(dst) = p.out_signed ? pool_pairs<true>(r0.x, r0.y, r1.x, r1.y) : pool_pairs<false>(r0.x, r0.y, r1.x, r1.y);
            } else {
                int a0 = src[0], a1 = src[1], c0 = src[p.WTP], c1 = src[p.WTP + 1];
                if (!p.out_signed) { a0 &= 0xFF; a1 &= 0xFF; c0 &= 0xFF; c1 &= 0xFF; }
                *dst = (int8_t)max(max(a0, a1), max(c0, c1));
            }
        }
    }
}

// Tile shape of one candidate and its modelled cost.
struct TileChoice {
    int TNX, TMX, TR, NSEG, XO, XB;
    double cost;
};

// Chooses channels per CTA (TNX * TN), rows per CTA (TR) and row segments so that the device is
// evenly loaded.  The model charges each "wave" of resident CTAs max(resident threads, 256) per SM
// (an SM with fewer threads than that cannot fill the multiply pipe), adds the staging work of a
// tile relative to its multiply work, and divides by the useful work.
static TileChoice choose_tiles(int total_rows, int Ho, int X, int K, int Co, int sms, int force_tr, bool even_rows, int xo_mult, int force_tnx) {
    constexpr int TM = kUTM, TN = kUTN;
    const int J = K;                                               // one tap per word
    TileChoice best;
    best.cost = -1.0;
    // More than four channel lanes (16 channels per CTA) never measured faster than four on the benchmark layers
    // (sweeps over every TNX and tile height: 10x20 to 160x320 maps, 3 to 256 input channels); the automatic choice
    // stays within 1 .. 4, a forced value may go up to 16.
    for (int TNX = 1; TNX <= (force_tnx > 0 ? 16 : 4); TNX *= 2) {
        if (force_tnx > 0 && TNX != force_tnx) continue;
        const int TCO = TNX * TN;
        if (TNX > 1 && TCO / 2 >= Co) break;                       // more channel lanes than channels
        const int gy = ceil_div(Co, TCO);
        const int max_tmx = kUThreads / TNX;
        const int maxpos = max_tmx * TM;
        // rows wider than a tile are cut into segments of XO blocks (a multiple of 4, so that every tile
        // row starts on a 16-byte boundary of the packed activations), each with its own J halo positions
        const int rowmax = std::min(maxpos, 64);                  // a staged row holds at most 64 words
        int NSEG = 1, XO = X;
        if (X + J > rowmax) {
            // xo_mult: a multiple of 4 (16-byte pieces of the packed rows); larger when the segments of a dense output
            // row have to start on byte boundaries
            XO = (rowmax - J) / xo_mult * xo_mult;
            if (XO < xo_mult) continue;
            NSEG = ceil_div(X, XO);
            XO = std::min(XO, (ceil_div(X, NSEG) + xo_mult - 1) / xo_mult * xo_mult);
            NSEG = ceil_div(X, XO);
        }
        const int XB = XO + J;
        const int tr_hi = std::max(1, std::min(maxpos / XB, total_rows));
        const int tr_lo = force_tr > 0 ? std::min(force_tr, tr_hi) : 1;
        const int tr_end = force_tr > 0 ? tr_lo : tr_hi;
        for (int TR = tr_lo; TR <= tr_end; ++TR) {
            if (even_rows && (TR & 1)) continue;                      // a fused 2x2 pool needs both rows of a pair in one CTA
            int TMX = ceil_div(TR * XB, TM);
            int threads = (TMX * TNX + 31) / 32 * 32;               // whole warps
            if (threads > kUThreads) continue;
            TMX = threads / TNX;
            const long long tiles = (long long)ceil_div(total_rows, TR) * NSEG * gy;
            // shared memory of the two double-buffered tiles (8 channels per stage at most)
            const int pitch = XB <= 8 ? 8 : XB <= 16 ? 16 : XB <= 32 ? 32 : 64;
            const int span_s = (TR + Ho - 2) / Ho + 1;
            const int ckc = stage_channel_cap(K, J);
            const size_t smem = 2 * 4 * ((size_t)ckc * ((TR + (K - 1) * span_s) * pitch + 8) + (size_t)ckc * K * J * kBPitch);
            if (smem > 72 * 1024) continue;                            // plus the second accumulators, 136 bytes per thread
            // (the model keeps charging 32 KB for them: with their true size it preferred tiles that measured slower)
            const int per_sm = std::max(1, std::min(std::min(2048 / threads, 65536 / (threads * 128)), (int)(220 * 1024 / (smem + 32 * 1024))));
            const long long slots = (long long)per_sm * sms;
            const long long full_waves = tiles / slots;
            const long long rest = tiles - full_waves * slots;
            double time = (double)full_waves * std::max(per_sm * threads, 256);
            if (rest > 0) time += std::max((int)((rest + sms - 1) / sms) * threads, 256);
            const int span = (TR + Ho - 2) / Ho + 1;
            const double NR = TR + (K - 1) * span;
            const double work = (double)K * J * (TM * TN + 8) * threads;
            const double stage = 0.5 * NR * XB + 0.5 * K * J * TCO;   // a few instructions per 16-byte piece
            time *= 1.0 + stage / work;
            const double useful = (double)total_rows * X * Co;     // output blocks x channels
            const double cost = time * sms / useful;
            if (best.cost < 0 || cost < best.cost - 1e-12) best = {TNX, TMX, TR, NSEG, XO, XB, cost};
        }
    }
    return best;
}

int setup_unpacked(int B, int Ci, int H, int W, int Co, int K, int pad, const OutputSpec &out, const hikonv_tuning_t *tune, int sms,
                   UnpackedLaunch *u) {
    if (K > kMaxJ) return HIKONV_ERR_UNSUPPORTED;
    UnpackedParams &p = u->p;
    std::memset(&p, 0, sizeof(p));
    const int Ho = H + 2 * pad - K + 1, Wo = W + 2 * pad - K + 1;
    p.B = B; p.Ci = Ci; p.Co = Co; p.CoP = (Co + 3) / 4 * 4; p.K = K; p.Ho = Ho; p.Wo = Wo; p.Hp = Ho + K - 1;
    p.requant = out.requant ? 1 : 0; p.shift = out.shift; p.lo = out.lo; p.hi = out.hi;
    p.total_rows = B * Ho;
    p.X = Wo;
    // tune->tile > 0: rows per CTA, plus 1000 x channel lanes per CTA (1, 2, 4, 8, 16) when those are forced too
    const int tile_arg = (tune && tune->tile > 0) ? tune->tile % 100000 : 0;
    const TileChoice tc = choose_tiles(p.total_rows, Ho, p.X, K, Co, sms, tile_arg % 1000, out.requant && out.pool,
                                       segment_multiple(out, 1), tile_arg / 1000);
    if (tc.cost < 0) return HIKONV_ERR_UNSUPPORTED;
    p.TNX = tc.TNX; p.TMX = tc.TMX; p.TCO = tc.TNX * kUTN;
    p.NSEG = tc.NSEG; p.XO = tc.XO; p.XB = tc.XB; p.TR = tc.TR;
    u->threads = tc.TMX * tc.TNX;
    const int span = (p.TR + Ho - 2) / Ho + 1;              // images a tile can touch
    // output offsets relative to a CTA's first image and channel are kept in 32 bits
    if ((double)(span + 1) * std::max(Co, p.TCO) * Ho * Wo >= 4294967296.0) return HIKONV_ERR_UNSUPPORTED;
    // words per row in shared memory: 8, 16, 32 or 64 (the unrolled kernels have them as constants)
    p.XBS = p.XB <= 8 ? 8 : p.XB <= 16 ? 16 : p.XB <= 32 ? 32 : 64;
    p.XBT = (p.NSEG - 1) * p.XO + (p.XB + 3) / 4 * 4;
    p.lead = (K + 3) / 4 * 4;                               // room for the xb - j reads in front of the first row
    p.a_plane = (p.TR + (K - 1) * span) * p.XBS + p.lead;
    p.CK = std::min(stage_channel_cap(K, K), Ci);
    auto magic = [](int d) -> uint32_t { return d <= 1 ? 0u : (uint32_t)((0x100000000ull + (unsigned)d - 1) / (unsigned)d); };
    p.mg_xb = magic(p.XB); p.mg_ho = magic(Ho); p.mg_xq = magic((p.XB + 3) / 4); p.mg_ck = magic(p.CK);
    p.a_words = p.CK * p.a_plane;
    p.b_off = 2 * p.a_words;
    p.b_words = p.CK * K * K * kBPitch;
    size_t words = (size_t)p.b_off + 2 * (size_t)p.b_words;
    const int rc = output_staging(out, Ho, Wo, p.NSEG, p.XO, &p.stage_out, &p.vec);
    if (rc != HIKONV_OK) return rc;
    p.pool = out.pool ? 1 : 0; p.out_signed = out.lo < 0 ? 1 : 0; p.out_bits = out.out_bits;
    p.WTP = (p.XO + 15) / 16 * 16;
    if (p.stage_out) words = std::max(words, (size_t)p.TCO * p.TR * p.WTP / 4);
    u->smem_bytes = words * 4 + 16;
    if (u->smem_bytes > 200 * 1024) return HIKONV_ERR_UNSUPPORTED;
    const long long gx = ((long long)p.total_rows + p.TR - 1) / p.TR * p.NSEG;
    const int gy = ceil_div(Co, p.TCO);
    if (gx > 0x7FFFFFFFLL || gy > 65535) return HIKONV_ERR_UNSUPPORTED;
    u->grid = dim3((unsigned)gx, (unsigned)gy, 1);
    return HIKONV_OK;
}

template <int KT, int PITCH>
static int launch_pitch(const UnpackedLaunch &u, cudaStream_t st) {
    auto kern = conv2d_unpacked_kernel<KT, PITCH>;
    return with_dynamic_smem(reinterpret_cast<const void *>(kern), u.smem_bytes,
                             [&] { return launch_dependent(kern, u.grid, dim3(u.threads), u.smem_bytes, st, u.p); });
}

template <int KT>
static int launch_kernel_size(const UnpackedLaunch &u, cudaStream_t st) {
    switch (u.p.XBS) {
        case 8: return launch_pitch<KT, 8>(u, st);
        case 16: return launch_pitch<KT, 16>(u, st);
        case 32: return launch_pitch<KT, 32>(u, st);
        default: return launch_pitch<KT, 64>(u, st);
    }
}

int launch_unpacked2d(const UnpackedLaunch &u, cudaStream_t st) {
    if (u.p.K == 3) return launch_kernel_size<3>(u, st);
    if (u.p.K == 1) return launch_kernel_size<1>(u, st);
    return launch_pitch<0, 0>(u, st);
}

}  // namespace hikonv
