"""3x3 layers whose words hold the weights of three filters (forced with tile = -3, or chosen for large first layers), against the oracle
and the kernel on words of pixels and taps (tile = -1)."""
import numpy as np
import pytest
import torch

from oracle import direct
from paper_2208_00763_b200 import binding as hk
from paper_2208_00763_b200 import inputs

from gpu_util import assert_exact, dev

pytestmark = pytest.mark.gpu


def _forced(B, Ci, H, W, Co, pad, p, q, xs, ws):
    return hk.conv2d_launches(B, Ci, H, W, Co, 3, pad, p, q, xs, ws, tune={"tile": -3}) == (1, 1)


# odd and even maps (a thread owns 2 x 2 pixels), rows of several segments, tiles across images, channels that fill words (of three) and
# groups of words unevenly, one and several steps of input channels, every width whose sums fit 17 bits
@pytest.mark.parametrize("layer", [(2, 3, 9, 21, 16, 1), (1, 1, 1, 1, 1, 1), (3, 2, 7, 131, 5, 0), (5, 3, 2, 6, 40, 2), (1, 3, 34, 700, 19, 1), (40, 3, 12, 20, 17, 1)])
@pytest.mark.parametrize("p, q, xs, ws", [(8, 4, False, True), (8, 4, True, False), (6, 6, True, True), (4, 4, False, False), (1, 2, False, True)])
def test_layers_on_words_of_three_filters(layer, p, q, xs, ws):
    B, Ci, H, W, Co, pad = layer
    assert _forced(B, Ci, H, W, Co, pad, p, q, xs, ws)
    x, w = inputs.conv2d_case(B, Ci, H, W, Co, 3, p, q, xs, ws, seed=11 + H + p)
    ref = direct.conv2d_nchw(x, w, pad)
    d_x, d_w = dev(x), dev(w)
    assert_exact(hk.conv2d(d_x, d_w, pad, p, q, xs, ws, tune={"tile": -3}), ref, "sums")
    for rq in ((p, 0, 15), (2, -100, 200)):
        want = direct.requant(ref, *rq)
        got = hk.conv2d(d_x, d_w, pad, p, q, xs, ws, requant=rq, tune={"tile": -3})
        assert_exact(got, hk.conv2d(d_x, d_w, pad, p, q, xs, ws, requant=rq, tune={"tile": -1}).cpu().numpy(), "codes %s" % (rq,))
        if rq[2] <= 127:
            assert_exact(got, want, "codes against the oracle")
        if ref.shape[2] % 2 == 0 and ref.shape[3] % 2 == 0:
            pooled = [hk.conv2d_dense(d_x.reshape(-1), x.shape, 8, d_w.reshape(-1), w.shape, 8, pad, p, q, xs, ws, requant=rq, pool=True,
                                      tune={"tile": t}) for t in (-3, -1)]
            assert torch.equal(*pooled), "pooled codes %s" % (rq,)


def test_many_input_channels_in_steps_and_extreme_codes():
    for x, w in inputs.extreme_2d(2, 60, 10, 37, 8, 3, 4, 4, False, True):
        assert _forced(2, 60, 10, 37, 8, 1, 4, 4, False, True)
        assert_exact(hk.conv2d(dev(x), dev(w), 1, 4, 4, False, True, tune={"tile": -3}), direct.conv2d_nchw(x, w, 1), "60 channels")
    for x, w in inputs.extreme_2d(3, 3, 11, 10, 7, 3, 8, 4, False, True):
        assert_exact(hk.conv2d(dev(x), dev(w), 1, 8, 4, False, True, tune={"tile": -3}), direct.conv2d_nchw(x, w, 1), "image")
    assert not _forced(64, 4, 160, 320, 16, 1, 8, 4, False, True)      # 4 x 9 products of 12 bits do not fit a slot


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_unaligned_tensors(shift):
    # inputs and outputs that begin at any byte, sizes that end at any byte
    x, w = inputs.conv2d_case(3, 3, 7, 13, 10, 3, 8, 4, False, True, seed=5)
    buf = torch.zeros(x.size + 8, dtype=torch.int8, device="cuda")
    buf[shift:shift + x.size] = dev(x).reshape(-1)
    out = torch.zeros(3 * 10 * 7 * 13 + 8, dtype=torch.int8, device="cuda")
    view = out[shift:shift + 3 * 10 * 7 * 13].reshape(3, 10, 7, 13)
    hk.conv2d(buf[shift:shift + x.size].reshape(x.shape), dev(w), 1, 8, 4, False, True, requant=(8, 0, 15), out=view, tune={"tile": -3})
    want = direct.requant(direct.conv2d_nchw(x, w, 1), 8, 0, 15)
    assert np.array_equal(view.cpu().numpy().astype(np.int64), want)
    assert int(out[:shift].abs().sum()) == 0 and int(out[shift + want.size:].abs().sum()) == 0


def test_large_first_layers_take_it_and_small_ones_do_not():
    assert hk.conv2d_launches(64, 3, 160, 320, 16, 3, 1, 8, 4, False, True, requant=True, pool=True) == (1, 1)
    assert hk.conv2d_launches(64, 3, 160, 320, 16, 3, 1, 8, 4, False, True, tune={"tile": -1})[0] == 2
    assert hk.conv2d_launches(64, 3, 160, 320, 16, 3, 1, 4, 4, False, True)[0] == 2                # nine products in a wide multiplication
    x, w = inputs.conv2d_case(8, 3, 160, 320, 16, 3, 8, 4, False, True, seed=9)
    assert hk.conv2d_launches(8, 3, 160, 320, 16, 3, 1, 8, 4, False, True, requant=True, pool=True) == (1, 1)
    got = hk.conv2d_dense(dev(x).reshape(-1), x.shape, 8, dev(w).reshape(-1), w.shape, 8, 1, 8, 4, False, True, requant=(8, 0, 15), pool=True)
    assert_exact(got, direct.maxpool2x2(direct.requant(direct.conv2d_nchw(x, w, 1), 8, 0, 15)), "eight images")
