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
    return hk.conv2d_form(B, Ci, H, W, Co, 3, pad, p, q, xs, ws, tune={"tile": -3})["form"] == hk.FORM_FILTERS


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
    assert _forced(3, 3, 11, 10, 7, 1, 8, 4, False, True)
    for x, w in inputs.extreme_2d(3, 3, 11, 10, 7, 3, 8, 4, False, True):
        assert_exact(hk.conv2d(dev(x), dev(w), 1, 8, 4, False, True, tune={"tile": -3}), direct.conv2d_nchw(x, w, 1), "image")
    assert not _forced(64, 4, 160, 320, 16, 1, 8, 4, False, True)      # 4 x 9 products of 12 bits do not fit a slot


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_unaligned_tensors(shift):
    # inputs and outputs that begin at any byte, sizes that end at any byte
    assert _forced(3, 3, 7, 13, 10, 1, 8, 4, False, True)
    x, w = inputs.conv2d_case(3, 3, 7, 13, 10, 3, 8, 4, False, True, seed=5)
    buf = torch.zeros(x.size + 8, dtype=torch.int8, device="cuda")
    buf[shift:shift + x.size] = dev(x).reshape(-1)
    out = torch.zeros(3 * 10 * 7 * 13 + 8, dtype=torch.int8, device="cuda")
    view = out[shift:shift + 3 * 10 * 7 * 13].reshape(3, 10, 7, 13)
    hk.conv2d(buf[shift:shift + x.size].reshape(x.shape), dev(w), 1, 8, 4, False, True, requant=(8, 0, 15), out=view, tune={"tile": -3})
    want = direct.requant(direct.conv2d_nchw(x, w, 1), 8, 0, 15)
    assert np.array_equal(view.cpu().numpy().astype(np.int64), want)
    assert int(out[:shift].abs().sum()) == 0 and int(out[shift + want.size:].abs().sum()) == 0


@pytest.mark.parametrize("at_x", [0, 1, 3])
def test_unaligned_tensors_of_whole_words(at_x):
    # a number of codes that is a multiple of four (the aligned input is read by words only), rows that can be stored in pairs: outputs at
    # any byte (codes) and at four bytes past a multiple of eight (sums) fall back to single stores
    B, Ci, H, W, Co = 4, 3, 8, 12, 10
    assert _forced(B, Ci, H, W, Co, 1, 8, 4, False, True)
    x, w = inputs.conv2d_case(B, Ci, H, W, Co, 3, 8, 4, False, True, seed=6)
    sums = direct.conv2d_nchw(x, w, 1)
    codes = direct.requant(sums, 8, 0, 15)
    buf = torch.zeros(x.size + 8, dtype=torch.int8, device="cuda")
    d_x = buf[at_x:at_x + x.size].copy_(dev(x).reshape(-1)).reshape(x.shape)
    for at, count, want, pool, dtype in ((0, sums.size, sums, 0, torch.int32), (1, sums.size, sums, 0, torch.int32), (1, codes.size, codes, 0, torch.int8),
                                         (2, codes.size, codes, 0, torch.int8), (3, codes.size // 4, direct.maxpool2x2(codes), 1, torch.int8)):
        out = torch.full((count + 8,), 77, dtype=dtype, device="cuda")
        hk.conv2d_dense(d_x.reshape(-1), x.shape, 8, dev(w).reshape(-1), w.shape, 8, 1, 8, 4, False, True, requant=(8, 0, 15) if dtype == torch.int8 else None,
                        out_store_bits=8, pool=bool(pool), out=out[at:at + count].reshape(want.shape), tune={"tile": -3})
        assert_exact(out[at:at + count].reshape(want.shape), want, "output %d past its alignment" % at)
        assert bool((out[:at] == 77).all()) and bool((out[at + count:] == 77).all())


# every instantiation of the kernel, with several steps of input channels and several tiles per CTA together, cut rows among them, signed and
# unsigned, aligned and unaligned tensors; pools of codes from below 0 to above 127 wrap
@pytest.mark.parametrize("words", [2, 4, 6])
@pytest.mark.parametrize("layer, groups, step, ctas", [((3, 3, 8, 530, 19, 1), 1, 2, 3), ((40, 5, 10, 18, 23, 0), 2, 2, 4), ((2, 6, 6, 300, 60, 1), 4, 1, 2),
                                                          ((2, 4, 40, 34, 17, 2), 1, 3, 1)])
@pytest.mark.parametrize("p, q, xs, ws, at", [(6, 4, False, True, 0), (5, 5, True, True, 1), (7, 2, True, False, 2), (4, 4, False, False, 0)])
def test_steps_and_tiles_of_every_instantiation(words, layer, groups, step, ctas, p, q, xs, ws, at):
    B, Ci, H, W, Co, pad = layer
    tune = {"tile": -(3 + 10 * words + 100 * groups + 1000 * step + 100000 * ctas)}
    x, w = inputs.conv2d_case(B, Ci, H, W, Co, 3, p, q, xs, ws, seed=21 + H + p)
    buf = torch.zeros(x.size + 8, dtype=torch.int8, device="cuda")
    d_x, d_w = buf[at:at + x.size].copy_(dev(x).reshape(-1)), dev(w).reshape(-1)
    sums = direct.conv2d_nchw(x, w, pad)
    for rq, pool in ((None, False), ((3, 0, 15), False), ((3, 0, 15), True), ((1, -100, 200), True)):
        form = hk.conv2d_form(B, Ci, H, W, Co, 3, pad, p, q, xs, ws, requant=rq is not None, pool=pool, tune=tune)
        assert form["form"] == hk.FORM_FILTERS and (form["words"], form["groups"], form["step_channels"]) == (words, groups, step), form
        assert form["ctas"] <= ctas and form["tiles"] >= 2 * form["ctas"] and (W < 300 or form["segments"] > 1), form
        if pool and (sums.shape[2] % 2 or sums.shape[3] % 2):
            continue
        got = hk.conv2d_dense(d_x, x.shape, 8, d_w, w.shape, 8, pad, p, q, xs, ws, requant=rq, pool=pool, tune=tune)
        if rq is None:
            want = sums
        else:
            want = direct.requant(sums, *rq)
            if rq[2] > 127:                                    # the stored bytes, as the layer's output is read back
                want = want.astype(np.int8).astype(np.int64)
            want = direct.maxpool2x2(want) if pool else want
        assert_exact(got, want, "%s words=%d requant=%s pool=%s" % (layer, words, rq, pool))


@pytest.mark.parametrize("layer, p, q, xs, words", [((4, 3, 112, 112, 20), 8, 4, False, 4), ((4, 3, 120, 112, 24), 8, 4, False, None), ((2, 6, 80, 80, 96), 6, 6, True, None),
                                                    ((700, 1, 10, 10, 16), 8, 4, False, None), ((23, 3, 32, 40, 64), 5, 7, True, None)])
def test_layers_that_take_it_by_themselves(layer, p, q, xs, words):
    B, Ci, H, W, Co = layer
    form = hk.conv2d_form(B, Ci, H, W, Co, 3, 1, p, q, xs, True, requant=True, pool=True)
    assert form["form"] == hk.FORM_FILTERS and (words is None or form["words"] == words), form
    x, w = inputs.conv2d_case(B, Ci, H, W, Co, 3, p, q, xs, True, seed=31 + H)
    sums = direct.conv2d_nchw(x, w, 1)
    got = hk.conv2d_dense(dev(x).reshape(-1), x.shape, 8, dev(w).reshape(-1), w.shape, 8, 1, p, q, xs, True, requant=(p + q - 5, 0, 15), pool=True)
    assert_exact(got, direct.maxpool2x2(direct.requant(sums, p + q - 5, 0, 15)), "%s" % (layer,))


def test_large_first_layers_take_it_and_small_ones_do_not():
    assert hk.conv2d_launches(64, 3, 160, 320, 16, 3, 1, 8, 4, False, True, requant=True, pool=True) == (1, 1)
    assert hk.conv2d_launches(64, 3, 160, 320, 16, 3, 1, 8, 4, False, True, tune={"tile": -1})[0] == 2
    assert hk.conv2d_launches(64, 3, 160, 320, 16, 3, 1, 4, 4, False, True)[0] == 2                # nine products in a wide multiplication
    x, w = inputs.conv2d_case(8, 3, 160, 320, 16, 3, 8, 4, False, True, seed=9)
    assert hk.conv2d_launches(8, 3, 160, 320, 16, 3, 1, 8, 4, False, True, requant=True, pool=True) == (1, 1)
    got = hk.conv2d_dense(dev(x).reshape(-1), x.shape, 8, dev(w).reshape(-1), w.shape, 8, 1, 8, 4, False, True, requant=(8, 0, 15), pool=True)
    assert_exact(got, direct.maxpool2x2(direct.requant(direct.conv2d_nchw(x, w, 1), 8, 0, 15)), "eight images")
