"""Three-dimensional layers around the lines where the forward splits a position's taps over threads and the
parameter gradients split their items: channel groups with a remainder, windows of one plane, windows too large
for whole groups, one channel and one plane (no split), a position count one past a block."""
import pytest

from paper_2504_06881_b200 import inputs
from test_gpu_3d import MODES, check

pytestmark = pytest.mark.gpu

L = inputs.layer3d
LAYERS = [
    L(1, 7, 5, 5, 5, 5, T=5, R=5, S=5),                       # one position, 7 channels x 5 planes over 32 slots
    L(3, 33, 4, 4, 5, 6, T=2, R=2, S=2),                      # channel groups with a remainder
    L(1, 9, 1, 12, 13, 9, T=1, R=7, S=7, pad=(0, 3, 3)),      # one plane
    L(2, 5, 8, 9, 9, 4, T=8, R=6, S=5, pad=(2, 1, 1)),        # 240 taps: small groups
    L(1, 1, 1, 9, 13, 3, T=1, R=3, S=3),                      # one channel and plane
    L(1, 2, 3, 5, 15, 3, T=3, R=3, S=3),                      # 39 positions
    L(2, 3, 9, 11, 10, 8, T=3, R=3, S=3, stride=(2, 3, 2), pad=1, dil=(1, 2, 1)),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode,chan", MODES)
def test_split_layers(mode, chan, dtype):
    for i, d in enumerate(LAYERS):
        check(dict(d, mode=mode, chan=chan, dtype=dtype), 1800 + i)
