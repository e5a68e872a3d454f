"""Backward of the Max / Min combine at the sizes where its tiles and classes change: rows and columns that
share input elements for strides and dilations, rows narrower than a warp (several to a warp) and wider, tiles
along the columns of a long row, more channels than one tile holds, output channels around 32, planes whose
pixels load one or four at a time."""
import pytest

from paper_2504_06881_b200 import inputs
import parity

pytestmark = pytest.mark.gpu

L = inputs.layer
LAYERS = [
    L(2, 3, 9, 9, 33, pad=1),                            # three rows to a warp, single pixels, K one past 32
    L(1, 2, 40, 32, 8, pad=1),                           # a warp's width, four pixels at a time
    L(1, 2, 21, 37, 9, pad=2, dil=2),                    # ... and past it; dilation: neighbours share a class
    L(2, 2, 23, 33, 6, stride=2, pad=1),
    L(1, 3, 19, 26, 5, stride=3, pad=2, dil=4),          # stride and dilation without a common step
    L(1, 2, 20, 24, 5, R=5, S=5, pad=2),
    L(1, 2, 3, 900, 7, R=3, S=3, pad=1),                 # column tiles
    L(2, 3, 1, 2500, 4, R=1, S=9, pad=(0, 4)),
    L(1, 2, 1, 1201, 3, R=1, S=5, pad=(0, 8), dil=4, stride=2),
    L(4, 3, 7, 7, 2, stride=4),                          # windows that share nothing
    L(1, 1, 1, 1, 1, R=1, S=1),
    L(1, 300, 12, 12, 3, pad=1),                         # channel blocks in both kernels
    L(1, 2, 30, 9, 3, pad=(5, 4)),                       # windows wholly inside the padding
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode,chan", [("max_plus", "max"), ("min_plus", "max"), ("max_plus", "min")])
def test_classes_and_tiles(mode, chan, dtype):
    for i, d in enumerate(LAYERS):
        parity.check_layer(dict(d, mode=mode, chan=chan, dtype=dtype), None, 2400 + i, recompute=False)


ODD = [
    L(3, 2, 9, 7, 33, pad=1),                            # rows that start at odd elements, the last at the tensor's end
    L(1, 1, 5, 5, 1, pad=1),
    L(5, 70, 15, 15, 40, pad=1),                         # several tiles of a plane, channel blocks
    L(2, 3, 11, 13, 3, pad=1),                           # lanes of one channel on several pixel slices
    L(3, 2, 7, 10, 5, pad=1),                            # an even plane that is not a multiple of four
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_odd_planes(dtype):
    for i, d in enumerate(ODD):
        parity.check_layer(dict(d, mode="max_plus", dtype=dtype), None, 2500 + i, recompute=False)
