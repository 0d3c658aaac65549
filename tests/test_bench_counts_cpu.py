"""CPU check of what bench.py reports for the 2-D workloads: launches, kernels and multiplies of the forms that run, each kind against its own rate."""
import os
import sys

import numpy as np
import pytest

from paper_2208_00763_b200 import binding as hk
from paper_2208_00763_b200 import inputs

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def _network():
    ch = inputs.C5_CHANNELS
    layers = [{"w": np.zeros((ch[i + 1], ch[i], 3, 3)), "pad": 1, "pool": inputs.C5_POOL[i], "p": 8 if i == 0 else 4, "q": 4, "x_signed": False,
               "w_signed": True} for i in range(8)]
    return layers, np.zeros((inputs.C5_HEAD_CHANNELS, ch[8], 1, 1))


def test_network_counts_follow_the_forms():
    layers, head = _network()
    forms, macs, out = bench.network_forms(hk, layers, head, 64, 160, 320, hk.ALGO_PACKED32, [None] * 8)
    assert [f["form"] for f in forms] == [hk.FORM_FILTERS] + [hk.FORM_TWO_LAUNCHES] * 8 and sum(f["launches"] for f in forms) == 17
    assert forms[0]["multiplies"] == 0 and forms[0]["double_multiplies"] == 64 * 160 * 320 * 6 * 27
    assert forms[8]["multiplies"] == hk.conv2d_multiplies(64, 64, 10, 20, 36, 1, 0, 4, 4, False, True) and out == (10, 20)
    assert bench.kernels_of(hk, forms) == "1 x conv2d_filters_kernel, 8 x conv2d_strip_kernel (multiplies summed)"
    plain, same, _ = bench.network_forms(hk, layers, head, 64, 160, 320, hk.ALGO_UNPACKED_IMAD, [None] * 8)
    assert same == macs and sum(f["launches"] for f in plain) == 18 and not any(f["double_multiplies"] for f in plain)


def test_rooflines_rate_each_kind_of_multiply_by_itself():
    forms = [{"multiplies": 6e9, "double_multiplies": 0.0}, {"multiplies": 0.0, "double_multiplies": 8e9}]
    peak = {"packed": 10e12, "double": 20e12, "packed_measured": 9e12, "double_measured": 18e12}
    r = bench.alu_roofline(forms, 2.0, peak, "packed")
    assert r["frac"] == pytest.approx((6e9 / 9e12 + 8e9 / 18e12) / 2e-3) and r["frac_of_derived"] == pytest.approx((6e9 / 10e12 + 8e9 / 20e12) / 2e-3)
    assert r["achieved"] == pytest.approx(r["frac"] * r["peak"])
    only = bench.alu_roofline(forms[:1], 2.0, peak, "packed")
    assert only["peak"] == pytest.approx(9.0) and only["frac"] == pytest.approx(6e9 / 9e12 / 2e-3)
