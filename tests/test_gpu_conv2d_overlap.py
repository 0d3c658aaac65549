"""Layers that write over their own inputs: the forms in one launch read inputs while outputs are written, so such calls take two launches."""
import numpy as np
import pytest
import torch

from oracle import direct
from paper_2208_00763_b200 import binding as hk
from paper_2208_00763_b200 import inputs

from gpu_util import dev

pytestmark = pytest.mark.gpu


# a large pooled first layer (words of several filters), a small layer (operands packed by the layer kernel), one of two launches anyway
@pytest.mark.parametrize("layer, p, q, xs, pool", [((9, 3, 160, 320, 16), 8, 4, False, True), ((2, 24, 20, 20, 32), 4, 4, True, False),
                                                   ((4, 64, 30, 30, 64), 4, 4, False, False)])
@pytest.mark.parametrize("tile", [0, -2, -3])
def test_outputs_over_inputs(layer, p, q, xs, pool, tile):
    B, Ci, H, W, Co = layer
    x, w = inputs.conv2d_case(B, Ci, H, W, Co, 3, p, q, xs, True, seed=3)
    codes = direct.requant(direct.conv2d_nchw(x, w, 1), p, 0, 15)
    if pool:
        codes = direct.maxpool2x2(codes)
    n_x, n_w, n_out = x.size, w.size, codes.size
    tune = {"tile": tile} if tile else None
    form = hk.conv2d_form(B, Ci, H, W, Co, 3, 1, p, q, xs, True, requant=True, pool=pool, tune=tune)["form"]     # where nothing overlaps
    assert form == {(3, 0): hk.FORM_FILTERS, (3, -3): hk.FORM_FILTERS, (24, -2): hk.FORM_ONE_LAUNCH}.get((Ci, tile), form)
    # where the output begins relative to the activations (half-way through, at their last piece, in front of them), or over the weights
    for at_x, at_w, at_out in ((0, None, 0), (0, None, n_x // 512 * 256), (0, None, (n_x - 1) // 256 * 256), (n_out // 512 * 256, None, 0), (None, 0, 0)):
        buf = torch.zeros(max(n_x, n_w) + 2 * n_out, dtype=torch.int8, device="cuda")
        d_x, d_w = dev(x).reshape(-1), dev(w).reshape(-1)
        if at_x is not None:
            d_x = buf[at_x:at_x + n_x].copy_(d_x)
        if at_w is not None:
            d_w = buf[at_w:at_w + n_w].copy_(d_w)
        out = buf[at_out:at_out + n_out].reshape(codes.shape)
        if pool:
            hk.conv2d_dense(d_x, x.shape, 8, d_w, w.shape, 8, 1, p, q, xs, True, requant=(p, 0, 15), pool=True, out=out, tune=tune)
        else:
            hk.conv2d(d_x.reshape(x.shape), d_w.reshape(w.shape), 1, p, q, xs, True, requant=(p, 0, 15), out=out, tune=tune)
        assert np.array_equal(out.cpu().numpy().astype(np.int64), codes), (layer, at_x, at_w, at_out)
