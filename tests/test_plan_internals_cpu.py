"""CPU checks of planning functions that are not part of the C interface (compiled from the library's own source)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <initializer_list>
#include "hikonv_internal.h"
using namespace hikonv;
// Layers whose layout needs no moves, with slots made narrower than the planner's: either all channels fit, or the answer is 0.
int main() {
    long layouts = 0, zero = 0, wrong = 0;
    for (int p = 1; p <= 8; ++p)
        for (int q = 1; q <= 8; ++q)
            for (int sg = 0; sg < 4; ++sg)
                for (int K : {1, 3, 5})
                    for (int Ci : {1, 2, 7, 40}) {
                        hikonv_layout_t L;
                        if (make_layout(p, q, sg & 1, sg >> 1, K, 2, Ci * K, 30, nullptr, &L) != HIKONV_OK || L.M < Ci * K) continue;
                        for (int less = 0; less < 6 && L.S > 1; ++less, --L.S) {
                            const SplitConsts sc = make_split_consts(L, p, q, sg & 1, sg >> 1, K, L.M);
                            const int cf = move_period(L, sc, p, q, sg & 1, sg >> 1, K, Ci, true);
                            ++layouts;
                            zero += cf == 0;
                            wrong += cf != 0 && cf != Ci;
                        }
                    }
    std::printf("%ld %ld %ld\n", layouts, zero, wrong);
}
"""


def test_channels_between_moves_without_moves_are_all_or_none(tmp_path):
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(DRIVER)
    csrc = os.path.join(ROOT, "paper_2208_00763_b200", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-o", str(exe), str(src),
                    os.path.join(csrc, "hikonv_plan.cpp")], check=True)
    layouts, zero, wrong = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert layouts > 1000 and zero > 100 and wrong == 0, (layouts, zero, wrong)
