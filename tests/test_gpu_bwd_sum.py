"""Backward of the Sum forms at the sizes where its tiles, shares and tables change: one tile of exactly 256
quads and one quad more, tiles along both axes (regions that overlap in rows and columns), several images
per tile with a remainder, output channels around the staged 32, whole and partial rounds of quads, the
table over winner pairs and the one per branch, 16-bit codes."""
import pytest

from paper_2504_06881_b200 import inputs, tconv
import parity

pytestmark = pytest.mark.gpu

L = inputs.layer
LAYERS = [
    L(2, 2, 32, 32, 33, pad=1),                          # one tile of 256 quads, K one past the staged 32
    L(1, 2, 33, 32, 8, pad=1),                           # a row more: two tiles
    L(2, 1, 40, 72, 5, pad=1),                           # tiles along both axes
    L(1, 2, 37, 70, 9, pad=2, dil=2),                    # ... and ragged rows, overlapping by four
    L(1, 1, 41, 75, 3, pad=4, dil=4),
    L(2, 2, 75, 50, 6, stride=2, pad=1),                 # stride: input gaps between the taps
    L(37, 3, 7, 7, 40, pad=1),                           # several images per tile, the last tile short
    L(64, 2, 16, 16, 2, pad=1),                          # whole rounds of 32 quads, pair table
    L(1, 1, 1, 1, 1, R=1, S=1),
    L(3, 2, 1, 61, 7, R=1, S=3, pad=(0, 1)),
    L(2, 2, 20, 24, 5, R=5, S=5, pad=2),                 # 16-bit codes
    L(2, 3, 17, 18, 4, R=4, S=4, pad=1),                 # 16 taps: one table per branch
    L(1, 2, 30, 9, 3, pad=(5, 4)),                       # windows wholly inside the padding
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode,chan", [("compound", "sum"), ("parallel", "sum"), ("max_plus", "sum"), ("min_plus", "sum")])
def test_tiles_and_shares(mode, chan, dtype):
    for i, d in enumerate(LAYERS):
        parity.check_layer(dict(d, mode=mode, chan=chan, dtype=dtype), None, 1700 + i, recompute=False)
        assert tconv.tconv_last_kernel() == "bwd_sum"


@pytest.mark.parametrize("need", [("grad_x",), ("grad_alpha", "grad_beta"), ("grad_w", "grad_w2"), ("grad_bias",)])
def test_single_gradients(need):
    """Every gradient on its own equals the one of the full call."""
    d = L(3, 4, 20, 28, 12, pad=1, mode="parallel")
    t = inputs.draw(d, 1750)
    g, _, win = parity.check_forward(d, t)
    la = parity.layer_args(d, g)
    full = tconv.backward(d, g["x"], g["w"], g["g"], la["w2"], la["alpha"], la["beta"], win)
    part = tconv.backward(d, g["x"], g["w"], g["g"], la["w2"], la["alpha"], la["beta"], win, need=need)
    assert set(part) == set(need)
    for k in need:
        assert (part[k] == full[k]).all(), k


def test_more_rows_than_blocks_of_one_grid_axis():
    d = L(1, 1, 2_100_000, 4, 1, pad=1, mode="compound")
    parity.check_layer(d, None, 1760, recompute=False)
    assert tconv.tconv_last_kernel() == "bwd_sum"
