// The packed method on small layers in ONE launch.
//
// A layer of a few hundred output pixels is bound by latency: a packing launch of 3.5 us, then threads that walk all input
// channels one after the other while most SMs have nothing to do.  Here a CTA packs what it needs itself (activation rows and
// kernel rows, Eq. 5, from the codes into shared memory) and the CTAs of a cluster share the input channels of one output tile:
// each sums its own, splits its slots into 32-bit sums, and the cluster adds them through distributed shared memory, every CTA
// finishing the rows and channels that fall to it.  Tile, products, moves, overlap-add and slots are those of the strip
// kernel (hikonv_conv2d_strip.cuh) with 2 x 4 rows x channels per thread.
// The packing is repeated by every CTA that reads a row, and a cluster's sums cross the network between SMs, so larger layers
// are faster on two launches: plan_layer compares the modelled times.  Time of one against two launches, one call after the
// other in a graph: 5 -> 183 channels on five 7x46 maps 3.7 / 4.2 us, 64 -> 36 channels 1x1 on one 10x20 map 5.0 / 6.9, 64 -> 64
// channels 3x3 on one 10x20 map 6.65 / 6.67, on 64 of them 22.5 / 16.3; 119 -> 37 channels 5x5 8-bit on two 18x17 maps 22.2 / 20.6.
// (The layers of the compact CNN run in two launches for one image, too.)
#include <type_traits>

#include "hikonv_cuda.cuh"
#include "hikonv_conv2d_small.h"
#include "hikonv_conv2d_util.cuh"

namespace hikonv {

// Not the .aligned forms: those want all threads of a warp at the instruction together, and the code in front of both barriers has
// branches that the threads of a warp take apart (the words from another warp, the stores).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ int32_t load_cluster(uint32_t smem_addr, uint32_t rank) {
    uint32_t remote;
    int32_t v;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_addr), "r"(rank));
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(remote) : "memory");
    return v;
}

template <int N, int KT, int JT>
constexpr bool kSmallPackedAdd = strip_packed_add(N, KT, JT);

template <int N, int KT, int JT, bool SP>
__global__ void __launch_bounds__(kStripThreads, 2) conv2d_small_kernel(const __grid_constant__ SmallParams q) {
    constexpr int TM = kSmallTM, TN = kSmallTN, ROWS = TM + KT - 1, KJ = KT * JT;
    constexpr bool PACKED_ADD = kSmallPackedAdd<N, KT, JT>, UP = N > 1 && KT != 1;
    extern __shared__ __align__(16) uint32_t smem[];
    grid_dependency_release();
    const StripParams &p = q.s;
    const int tid = threadIdx.x, nthreads = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int tnx_log2 = 31 - __clz(p.TNX), tn = tid & (p.TNX - 1);
    const int rank = blockIdx.z;                               // of the CTA in its cluster
    const int g0 = blockIdx.x * p.TS, b0 = g0 / p.SH, s0 = g0 - b0 * p.SH, TSe = min(p.TS, p.strips - g0);
    const int co0 = blockIdx.y * p.TCO;
    const int r0 = s0 * TM;                                    // first staged row, in padded rows of image b0
    const int pos = tid >> tnx_log2, pos_ok = pos < TSe * p.XB, pc = pos_ok ? pos : 0;
    const int sl = fast_div(pc, p.mg_xb), xb = pc - sl * p.XB;
    const int db = fast_div(s0 + sl, p.mg_sh), s_img = s0 + sl - db * p.SH;
    const int c0 = rank * q.Cz, cn = min(q.Cz, p.Ci - c0);     // this CTA's input channels (none for the last CTAs of an uneven cut)

    grid_dependency_wait();                                    // the input may come from the kernel before
    // ---- pack the activation rows: [channel][row][word], 16 bytes at a time
    const int xq = p.pitch / 4;
    const uint32_t a_items = cn > 0 ? (uint32_t)(cn * q.rows * xq) : 0u;
    for (uint32_t i = tid; i < a_items; i += nthreads) {
        const int rest = fast_div((int)i, q.mg_xq), w4 = (int)i - rest * xq;
        const int c = fast_div(rest, q.mg_rows), r = rest - c * q.rows;
        const int d = fast_div(r0 + r, q.mg_hp), b = b0 + d, h = r0 + r - d * p.Hp - p.pad;
        uint32_t word[4] = {0u, 0u, 0u, 0u};
        const int col0 = q.col_first + 4 * w4 * N;
        const bool row_in = b < q.B && h >= 0 && h < q.H;
        if (row_in && col0 + 4 * N > 0 && col0 < p.W)
            pack_row_words<N>(q.x, ((b * p.Ci + c0 + c) * q.H + h) * p.W, q.ragged, p.W, col0, true, 0u, q.x_signed != 0, p.S, word);
        *reinterpret_cast<uint4 *>(smem + c * p.plane + r * p.pitch + 4 * w4) = make_uint4(word[0], word[1], word[2], word[3]);
    }
    // ---- pack the kernel rows of these input and output channels (reversed rows, Theorem 3): [(ci, kh, j)][channel]
    uint32_t *const Bs = smem + p.b_off;
    const int tco_log2 = 31 - __clz(p.TCO);
    for (int i = tid; i < (cn > 0 ? cn * KJ << tco_log2 : 0); i += nthreads) {
        const int rj = i >> tco_log2, c = i & (p.TCO - 1), row = rj / JT, j = rj - row * JT;
        uint32_t word = 0;
        if (co0 + c < p.Co) {
            const int8_t *src = q.w + ((size_t)(co0 + c) * p.Ci * KT + c0 * KT + row) * KT;
            int8_t code[KT];
#pragma unroll
            for (int k = 0; k < KT; ++k) code[k] = load_ordered(src + k);
#pragma unroll
            for (int g = 0; g < KT; ++g) {                     // tap g of the reversed row belongs to chunk g / Kc
                const int32_t v = q.w_signed ? (int32_t)code[KT - 1 - g] : (int32_t)(uint8_t)code[KT - 1 - g];
                const int slot = g - j * q.Kc;
                if (slot >= 0 && slot < q.Kc) word += (uint32_t)v << (p.S * slot);
            }
        }
        Bs[rj * kStripBPitch + c] = word;
    }
    __syncthreads();

    // ---- products of this CTA's channels
    uint64_t acc[TM][TN], e[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int t = 0; t < TN; ++t) {
            acc[i][t] = p.bias;
            e[i][t] = 0ull;
        }
    int a_off[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) a_off[r] = (db * p.Hp + (s_img - s0) * TM + r) * p.pitch + xb + JT - 1;
    int moves = 0, left = q.CF;
#pragma unroll 2
    for (int c = 0; c < cn; ++c) {
        const int a_ch = c * p.plane, b_ch = p.b_off + c * KJ * kStripBPitch + tn * TN;
        uint32_t a[ROWS][JT];
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int j = 0; j < JT; ++j) a[r][j] = smem[a_ch + a_off[r] - j];
#pragma unroll
        for (int kh = 0; kh < KT; ++kh)
#pragma unroll
            for (int j = 0; j < JT; ++j) {
                const uint4 v = *reinterpret_cast<const uint4 *>(smem + b_ch + (kh * JT + j) * kStripBPitch);
                const uint32_t b[TN] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int t = 0; t < TN; ++t) mad_wide<SP>(acc[i][t], a[i + kh][j], b[t]);
            }
        if (--left == 0 && c + 1 < cn) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int t = 0; t < TN; ++t) {
                    e[i][t] += (acc[i][t] >> p.h) & p.mask_high;
                    acc[i][t] = (acc[i][t] & p.mask_low) | p.bias;
                }
            ++moves;
            left = q.CF;
        }
    }

    // ---- words above the N low slots to the next lane, then the slots as 32-bit sums
    uint2 *xch = reinterpret_cast<uint2 *>(smem) + ((warp << tnx_log2) + tn) * (TM * TN);
    const int lanes_m = 32 >> tnx_log2, lm = lane >> tnx_log2;
    __syncthreads();
    if (UP && lm == lanes_m - 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int t = 0; t < TN; ++t) xch[i * TN + t] = make_uint2((uint32_t)(acc[i][t] >> p.SN), (uint32_t)(e[i][t] >> p.SN));
    }
    __syncthreads();
    const uint2 *xch_in = xch - p.TNX * (TM * TN);
    const bool from_smem = lm == 0 && warp > 0;
    const uint32_t keep = xb == 0 ? 0u : 0xFFFFFFFFu, mask = p.slot_mask;
    int32_t y[TM][TN][N];
#pragma unroll
    for (int t = 0; t < TN; ++t)
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            uint64_t qa = acc[i][t], ea = e[i][t];
            uint32_t q_in = 0, e_in = 0;
            if constexpr (UP) {
                q_in = __shfl_up_sync(0xFFFFFFFFu, (uint32_t)(qa >> p.SN), p.TNX);
                e_in = __shfl_up_sync(0xFFFFFFFFu, (uint32_t)(ea >> p.SN), p.TNX);
                if (from_smem) {
                    const uint2 v = xch_in[i * TN + t];
                    q_in = v.x;
                    e_in = v.y;
                }
                q_in &= keep;
                e_in &= keep;
            }
            if constexpr (PACKED_ADD && UP) {
                qa = (qa & 0xFFFFFFFF00000000ull) | (uint32_t)((uint32_t)qa + q_in);
                ea = (ea & 0xFFFFFFFF00000000ull) | (uint32_t)((uint32_t)ea + e_in);
            }
#pragma unroll
            for (int m = 0; m < N; ++m) {
                int32_t v = -(moves + 1) * (p.slot_bias[m] + (keep ? p.slot_bias[m + N] : 0));
                v += (int32_t)((uint32_t)(qa >> (p.S * m)) & mask) + (int32_t)(((uint32_t)(ea >> (p.S * m)) & mask) << p.h);
                if constexpr (!PACKED_ADD && UP) {
                    if (m < p.up_slots) v += (int32_t)((q_in >> (p.S * m)) & mask) + (int32_t)(((e_in >> (p.S * m)) & mask) << p.h);
                }
                y[i][t][m] = v;
            }
        }

    // ---- sum over the cluster: CTA `rank` finishes the (t, i) pairs u = 2 t + i with u >> (3 - ks_log2) == rank
    const int ks = 1 << q.ks_log2, share_log2 = 3 - q.ks_log2;
    int32_t *red = reinterpret_cast<int32_t *>(smem + q.red_off);
    if (ks > 1) {
#pragma unroll
        for (int u = 0; u < TM * TN; ++u)
#pragma unroll
            for (int m = 0; m < N; ++m) red[(u * N + m) * nthreads + tid] = y[u & 1][u >> 1][m];
        cluster_arrive();
        cluster_wait();
        const uint32_t mine = smem_address(red + tid);
#pragma unroll
        for (int u = 0; u < TM * TN; ++u)
            if ((u >> share_log2) == rank) {
#pragma unroll
                for (int m = 0; m < N; ++m) {
                    int32_t v = 0;
                    for (int z = 0; z < ks; ++z) v += load_cluster(mine + 4u * (uint32_t)((u * N + m) * nthreads), (uint32_t)z);
                    y[u & 1][u >> 1][m] = v;
                }
            }
        cluster_arrive();                                      // waited for at the end: no CTA leaves while its sums are read
    }

    const int w0 = xb * N - p.col_off, h0 = s_img * TM;
    bool col_ok[N];
#pragma unroll
    for (int m = 0; m < N; ++m) col_ok[m] = pos_ok && w0 + m >= 0 && w0 + m < p.Wo;
    auto requant = [&](int32_t v) { return max(p.lo, min(p.hi, v >> p.shift)); };
    if (!p.pool) {
        const size_t at = (((size_t)(b0 + db) * p.Co + co0 + tn * TN) * p.Ho + h0) * p.Wo + w0;
#pragma unroll
        for (int u = 0; u < TM * TN; ++u) {
            const int t = u >> 1, i = u & 1;
            if ((u >> share_log2) == rank && co0 + tn * TN + t < p.Co && h0 + i < p.Ho) {
                const size_t o = at + ((size_t)t * p.Ho + i) * p.Wo;
#pragma unroll
                for (int m = 0; m < N; ++m)
                    if (col_ok[m]) {
                        if (p.requant) ((int8_t *)p.out)[o + m] = (int8_t)requant(y[i][t][m]);
                        else ((int32_t *)p.out)[o + m] = y[i][t][m];
                    }
            }
        }
    } else {
        // the two rows of a pair are the thread's; neighbouring columns meet in shared memory
        int8_t *tile = reinterpret_cast<int8_t *>(smem + p.tile_off);
        const int tile_chan = p.TS * p.WTP;
#pragma unroll
        for (int t = 0; t < TN; ++t)
            if (((2 * t) >> share_log2) == rank) {
#pragma unroll
                for (int m = 0; m < N; ++m) {
                    // (codes from below 0 to above 127: the maximum of the bytes, as they are stored)
                    const int32_t v = p.pool == 2 ? max((int32_t)(int8_t)requant(y[0][t][m]), (int32_t)(int8_t)requant(y[1][t][m]))
                                                  : requant(max(y[0][t][m], y[1][t][m]));
                    if (col_ok[m]) tile[(tn * TN + t) * tile_chan + sl * p.WTP + w0 + m] = (int8_t)v;
                }
            }
        __syncthreads();
        const int nt_log2 = share_log2 - 1;                    // channels of a thread that this CTA finishes
        const int Hq = p.Ho >> 1, Wq = p.Wo >> 1, ch = p.TNX << nt_log2;
        const float inv_w = 1.0f / (float)Wq, inv_s = 1.0f / (float)TSe;
        for (int i = tid; i < ch * TSe * Wq; i += nthreads) {
            const int rest = small_div(i, Wq, inv_w), col = i - rest * Wq;
            const int k = small_div(rest, TSe, inv_s), ts = rest - k * TSe;
            const int cl = (k >> nt_log2) * TN + (rank << nt_log2) + (k & ((1 << nt_log2) - 1));
            const int d = fast_div(s0 + ts, p.mg_sh), hq = s0 + ts - d * p.SH;
            if (co0 + cl >= p.Co || hq >= Hq) continue;
            int a = tile[cl * tile_chan + ts * p.WTP + 2 * col], b = tile[cl * tile_chan + ts * p.WTP + 2 * col + 1];
            if (!p.out_signed) { a &= 0xFF; b &= 0xFF; }
            ((int8_t *)p.out)[(((size_t)(b0 + d) * p.Co + co0 + cl) * Hq + hq) * Wq + col] = (int8_t)max(a, b);
        }
    }
    if (ks > 1) cluster_wait();
}

template <int N, int KT, int JT>
static int launch_small_layout(const SmallLaunch &l, cudaStream_t st) {
    auto run = [&](auto kern) -> int {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = l.grid;
        cfg.blockDim = dim3(l.threads);
        cfg.dynamicSmemBytes = l.smem_bytes;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 1;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = l.grid.z;
        cfg.attrs = attr;
        cfg.numAttrs = l.grid.z > 1 ? 2 : 1;
        return with_dynamic_smem(reinterpret_cast<const void *>(kern), l.smem_bytes,
                                 [&] { return cudaLaunchKernelEx(&cfg, kern, l.p) == cudaSuccess ? HIKONV_OK : HIKONV_ERR_CUDA; });
    };
    return l.sp ? run(conv2d_small_kernel<N, KT, JT, true>) : run(conv2d_small_kernel<N, KT, JT, false>);
}

int launch_small(const SmallLaunch &l, int N, cudaStream_t st) {
    const int K = l.p.s.K, J = l.p.s.J;
#define HK_LAYOUT(n, k, j) if (N == n && K == k && J == j) return launch_small_layout<n, k, j>(l, st);
    HK_LAYOUT(2, 1, 1) HK_LAYOUT(3, 1, 1) HK_LAYOUT(4, 1, 1)
    HK_LAYOUT(2, 3, 1) HK_LAYOUT(2, 3, 2) HK_LAYOUT(3, 3, 1) HK_LAYOUT(4, 3, 1)
    HK_LAYOUT(2, 5, 3) HK_LAYOUT(3, 5, 2) HK_LAYOUT(4, 5, 1) HK_LAYOUT(4, 5, 2)
#undef HK_LAYOUT
    return HIKONV_ERR_UNSUPPORTED;
}

}  // namespace hikonv
