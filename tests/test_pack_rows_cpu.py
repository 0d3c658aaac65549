"""CPU check of the row packing of the 2-D kernels: the device function, compiled for the host with stand-ins for the device's
intrinsics, packs the words of Eq. 5 and reads no byte outside the caller's tensor, whatever its alignment and size."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
using std::max;
using std::min;
static const int8_t *g_lo, *g_hi;      // the tensor
static long g_outside = 0;
template <typename T> T __ldg(const T *p) {
    const int8_t *b = (const int8_t *)p;
    if (b < g_lo || b + sizeof(T) > g_hi) { ++g_outside; return T(0); }
    T v; std::memcpy(&v, b, sizeof(T)); return v;
}
static uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, int s) { return (uint32_t)((((uint64_t)hi << 32) | lo) >> (s & 31)); }
static uint32_t __vsub4(uint32_t a, uint32_t b) {
    uint32_t r = 0;
    for (int i = 0; i < 32; i += 8) r |= (((a >> i) - (b >> i)) & 0xFFu) << i;
    return r;
}
static uint32_t byte_permute(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r = 0;
    const uint64_t v = ((uint64_t)b << 32) | a;
    for (int i = 0; i < 4; ++i) {
        const uint32_t n = (sel >> (4 * i)) & 15u, byte = (uint32_t)(v >> (8 * (n & 7))) & 0xFFu;
        r |= ((n & 8) ? ((byte & 0x80u) ? 0xFFu : 0u) : byte) << (8 * i);
    }
    return r;
}
static uint32_t byte_range_mask(int i, int first, int last) {
    uint32_t m = 0;
    for (int b = 0; b < 4; ++b) if (4 * i + b >= first && 4 * i + b < last) m |= 0xFFu << (8 * b);
    return m;
}
template <typename T> T load_ordered(const T *p) { return __ldg(p); }
#define __host__
#define __device__
#define __forceinline__ inline
//FUNCTION
static long g_wrong = 0, g_words = 0;
template <int N> void sweep(int W, int rows, int shift, bool is_signed, int off, int S) {
    alignas(64) static int8_t buf[4096];
    int8_t *x = buf + 64 + shift;                       // buf + 64 is aligned
    const int n = W * rows;
    for (int i = 0; i < (int)sizeof(buf); ++i) buf[i] = (int8_t)(rand() & (is_signed ? 0x7F : 0x0F)) - (is_signed ? 64 : 0);
    g_lo = x; g_hi = x + n;
    for (int r = 0; r < rows; ++r)
        for (int in = 0; in < 2; ++in)
            for (int col0 = -2 * N; col0 < W; col0 += (rand() % 3) + 1) {
                if (col0 + 4 * N <= 0) continue;
                uint32_t word[4];
                pack_row_words<N>(x, r * W, ragged_codes(x, n), W, col0, in != 0, (uint32_t)off * 0x01010101u, is_signed || off != 0, S, word);
                for (int w = 0; w < 4; ++w, ++g_words) {
                    uint32_t want = 0;
                    for (int k = 0; k < N; ++k) {
                        const int c = col0 + w * N + k;
                        if (c < 0 || c >= W) continue;
                        const int v = (in ? (is_signed ? (int)x[r * W + c] : (int)(uint8_t)x[r * W + c]) : 0) - off;
                        want += (uint32_t)v << (S * k);
                    }
                    if (word[w] != want) ++g_wrong;
                }
            }
}
int main() {
    srand(5);
    for (int W = 1; W <= 23; ++W)
        for (int rows = 1; rows <= 3; ++rows)
            for (int shift = 0; shift < 4; ++shift) {
                sweep<1>(W, rows, shift, false, 0, 20); sweep<2>(W, rows, shift, true, 0, 13); sweep<2>(W, rows, shift, false, 8, 13);
                sweep<3>(W, rows, shift, false, 0, 10); sweep<4>(W, rows, shift, true, 0, 8); sweep<3>(W, rows, shift, false, 8, 10);
            }
    printf("%ld %ld %ld\n", g_words, g_wrong, g_outside);
}
"""


@pytest.fixture(scope="module")
def function_source():
    text = open(os.path.join(ROOT, "paper_2208_00763_b200", "csrc", "hikonv_conv2d_util.cuh")).read()
    parts = [re.search(pattern, text, re.S) for pattern in (r"__host__ inline int ragged_codes\(.*?\n",
                                                            r"template <int N>\n__device__ __forceinline__ void pack_row_words\(.*?\n}\n")]
    assert all(parts)
    return "".join(p.group(0) for p in parts)


def test_rows_are_packed_from_inside_the_tensor(function_source, tmp_path):
    src, exe = tmp_path / "harness.cpp", tmp_path / "harness"
    src.write_text(HARNESS.replace("//FUNCTION", function_source))
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wno-unknown-pragmas", "-o", str(exe), str(src)], check=True)
    words, wrong, outside = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert words > 50000 and wrong == 0 and outside == 0, (words, wrong, outside)
