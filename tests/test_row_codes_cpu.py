"""CPU check of how the 2-D kernel on words of several filters reads activations: the device function, compiled for the host, gives the
four codes of a row from any column on, reads nothing outside the caller's tensor, and reads single bytes only at its unaligned ends."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
static const int8_t *g_lo, *g_hi;      // the tensor
static long g_outside = 0, g_bytes = 0, g_loads = 0;
template <typename T> T load_ordered(const T *p) {
    const int8_t *b = (const int8_t *)p;
    ++g_loads;
    if (sizeof(T) == 1) ++g_bytes;
    // (an aligned tensor's words never reach outside it)
    if (b < g_lo || b + sizeof(T) > g_hi || (uintptr_t)b % sizeof(T) != 0) { ++g_outside; return T(0); }
    T v; std::memcpy(&v, b, sizeof(T)); return v;
}
#define __device__
#define __forceinline__ inline
//FUNCTION
int main() {
    long wrong = 0, codes = 0, most_bytes = 0;
    srand(7);
    for (int W = 1; W <= 19; ++W)
        for (int rows = 1; rows <= 6; ++rows)
            for (int shift = 0; shift < 4; ++shift) {
                alignas(64) static int8_t buf[512];
                int8_t *x = buf + 64 + shift;
                const int n = W * rows;
                for (int8_t &v : buf) v = (int8_t)rand();
                g_lo = x; g_hi = x + n; g_bytes = 0;
                for (int r = 0; r < rows; ++r)
                    for (int col0 = -9; col0 < W + 9; ++col0) {
                        uint32_t lo = 0, hi = 0, off = 0;
                        if (((uintptr_t)x | (unsigned)n) & 3) load_row_codes<true>(x, r * W, n, W, col0, lo, hi, off);
                        else load_row_codes<false>(x, r * W, n, W, col0, lo, hi, off);
                        const uint32_t v = off ? (uint32_t)((((uint64_t)hi << 32) | lo) >> (8 * off)) : lo;
                        for (int k = 0; k < 4; ++k, ++codes)
                            if (col0 + k >= 0 && col0 + k < W && (uint8_t)(v >> (8 * k)) != (uint8_t)x[r * W + col0 + k]) ++wrong;
                    }
                // seven columns reach the tensor's first word and seven its last one
                if (n >= 8 && g_bytes > most_bytes) most_bytes = g_bytes;
            }
    printf("%ld %ld %ld %ld %ld\n", codes, wrong, g_outside, g_loads, most_bytes);
}
"""


def test_row_codes_are_read_by_words_from_inside_the_tensor(tmp_path):
    text = open(os.path.join(ROOT, "paper_2208_00763_b200", "csrc", "hikonv_conv2d_filters.cu")).read()
    part = re.search(r"template <bool RAGGED>\n__device__ __forceinline__ void load_row_codes\(.*?\n}\n", text, re.S)
    assert part
    src, exe = tmp_path / "harness.cpp", tmp_path / "harness"
    src.write_text(HARNESS.replace("//FUNCTION", part.group(0)))
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", str(exe), str(src)], check=True)
    codes, wrong, outside, loads, most_bytes = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert codes > 100000 and wrong == 0 and outside == 0 and loads > 10000, (codes, wrong, outside, loads)
    assert most_bytes <= 2 * 7 * 3, most_bytes       # two end words of three codes at most, each read from seven columns
