"""CPU checks of the host query for the form a layer runs in: the rule for words of three filters, condition by condition, and the counts."""
import pytest

from paper_2208_00763_b200 import binding as hk

FIRST = dict(B=2, Ci=3, H=160, W=320, Co=16, K=3, pad=1, p=8, q=4, x_signed=False, w_signed=True, requant=True, pool=True)


def _form(**changes):
    return hk.conv2d_form(**{**FIRST, **changes})


@pytest.mark.parametrize("changes", [{}, {"Co": 20}, {"Ci": 6, "p": 6, "q": 6, "x_signed": True}, {"H": 32, "W": 32, "B": 100}, {"pad": 0, "B": 3}])
def test_pooled_first_layers_run_on_words_of_three_filters(changes):
    form = _form(**changes)
    layer = {**FIRST, **changes}
    rows, row = layer["H"] + 2 * layer["pad"] - 2, layer["W"] + 2 * layer["pad"] - 2
    assert form["form"] == hk.FORM_FILTERS and form["launches"] == 1 and form["cluster"] == 0 and form["multiplies"] == 0.0
    assert form["double_multiplies"] == layer["B"] * rows * row * -(-layer["Co"] // 3) * layer["Ci"] * 9
    assert form["words"] in (2, 4, 6) and form["ctas"] <= form["tiles"] and 1 <= form["step_channels"] <= layer["Ci"]
    launches, cluster = hk.conv2d_launches(**layer)
    assert launches == 1 and cluster == 1


@pytest.mark.parametrize("changes", [
    {"B": 1},                                                       # 0.8 million sums
    {"Co": 8, "B": 8},                                              # two of the words' three thirds for eight of nine filters
    {"pool": False}, {"requant": False, "pool": False},             # the other form stores directly
    {"Ci": 7, "p": 4, "q": 6}, {"Ci": 4},                           # more than six channels; sums beyond 17 bits
    {"p": 4},                                                       # more than three products in a word of pixels
    {"K": 5, "pad": 2}, {"K": 1, "pad": 0},
    {"tune": {"tile": -1}}, {"tune": {"N": 2}}, {"algo": hk.ALGO_UNPACKED_IMAD}])
def test_other_layers_do_not(changes):
    form = _form(**changes)
    assert form["form"] != hk.FORM_FILTERS and form["double_multiplies"] == 0.0 and form["multiplies"] > 0.0
    assert form["launches"] == (1 if form["form"] == hk.FORM_ONE_LAUNCH else 2)


@pytest.mark.parametrize("layer, p, q, xs", [((20, 4, 46, 80, 26), 5, 7, True), ((6, 6, 52, 120, 39), 7, 5, True), ((197, 5, 8, 86, 37), 4, 8, True),
                                             ((138, 4, 14, 56, 30), 7, 4, False), ((69, 6, 12, 90, 28), 5, 7, True), ((42, 6, 80, 34, 28), 8, 4, True)])
def test_tiles_that_do_not_stage_the_input_for_two_words_at_a_time(layer, p, q, xs):
    # with tiles of two words, every CTA row of which stages all activations again, these were 2 to 29 % slower than in two launches
    B, Ci, H, W, Co = layer
    form = hk.conv2d_form(B, Ci, H, W, Co, 3, 1, p, q, xs, True, requant=True, pool=True)
    assert form["form"] == hk.FORM_FILTERS and form["words"] * form["groups"] >= 4, form


def test_forced_parts_of_the_tile():
    for words in (2, 4, 6):
        for groups in (1, 2, 4):
            form = _form(Co=64, tune={"tile": -(3 + 10 * words + 100 * groups + 2000 + 900000)})
            assert form["form"] == hk.FORM_FILTERS and (form["words"], form["groups"], form["step_channels"]) == (words, groups, 2)
            assert form["ctas"] <= 9 and form["tiles"] > form["ctas"]
    # what does not fit is chosen automatically
    assert _form(tune={"tile": -13})["form"] == _form(pool=False, tune={"tile": -13})["form"] == hk.FORM_TWO_LAUNCHES
    assert _form(Ci=40, tune={"tile": -3})["form"] == hk.FORM_TWO_LAUNCHES


def test_counts_of_the_other_forms():
    layer = dict(B=1, Ci=24, H=20, W=20, Co=32, K=3, pad=1, p=4, q=4, x_signed=True, w_signed=True)
    two, one = hk.conv2d_form(**layer, tune={"tile": -1}), hk.conv2d_form(**layer, tune={"tile": -2})
    assert two["form"] == hk.FORM_TWO_LAUNCHES and two["multiplies"] == hk.conv2d_multiplies(**layer, tune={"tile": -1})
    # one word per N = 3 pixels of the row and its left edge, one chunk: 7 words a row
    assert one["form"] == hk.FORM_ONE_LAUNCH and one["cluster"] in (1, 2, 4, 8) and one["multiplies"] == 20 * 7 * 32 * 24 * 3
    assert hk.conv2d_form(**layer, algo=hk.ALGO_UNPACKED_IMAD)["form"] == hk.FORM_UNPACKED
