"""bf16 forward of 5x5 windows where its tiles end: one row and column of quads past a tile, output channels
around the eight (winners: four) of a thread, one input channel and an odd number of them, winners of 16 bits."""
import pytest

from paper_2504_06881_b200 import inputs, tconv
import parity

pytestmark = pytest.mark.gpu

L = inputs.layer
LAYERS = [
    L(2, 1, 28, 28, 6, R=5, S=5),                        # one input channel, K below the tile
    L(1, 3, 33, 36, 9, R=5, S=5, pad=2),                 # K one past eight, ragged rows
    L(2, 2, 17, 21, 33, R=5, S=5, pad=(2, 0)),           # K one past the tile, ragged columns
    L(1, 5, 5, 70, 4, R=5, S=5, pad=2),                  # wide rows, several column tiles
    L(3, 4, 5, 5, 3, R=5, S=5),                          # one output per image
]


@pytest.mark.parametrize("mode,chan", [("compound", "sum"), ("parallel", "sum"), ("max_plus", "sum"), ("min_plus", "sum"),
                                       ("max_plus", "max"), ("min_plus", "max"), ("max_plus", "min")])
def test_five_by_five(mode, chan):
    for i, d in enumerate(LAYERS):
        d = dict(d, mode=mode, chan=chan, dtype="bf16")
        t = inputs.draw(d, 2300 + i)
        parity.check_forward(d, t)
        tiled = chan == "sum" or d["C"] >= 5      # Max / Min winners of few channels: the any-shape kernel
        assert tconv.tconv_last_kernel().startswith("fwd_tiled_bf16" if tiled else "fwd_generic"), d
        parity.check_layer(d, None, 2300 + i, recompute=False)
