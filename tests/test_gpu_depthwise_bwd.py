"""All gradients of 3x3 stride-1 depthwise layers at the sizes where the strips of the backward change: one strip and
several, a short last strip, widths that are not whole quads, no padding and padding 2 (winners in the padding),
one image per chunk of the parameter sums and several."""
import pytest

from paper_2504_06881_b200 import inputs
from test_gpu_depthwise import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["compound", "parallel"])
def test_strips_and_borders(mode):
    mk = lambda N, C, H, W, pad: inputs.layer(N, C, H, W, C, 3, 3, mode=mode, pad=pad)
    cases = [mk(3, 4, 12, 12, 1), mk(2, 3, 37, 9, 1), mk(5, 2, 10, 10, 2), mk(2, 2, 13, 18, 0), mk(9, 160, 11, 14, 1),
             mk(1, 1, 45, 63, (2, 1)), mk(2, 1, 101, 4, 1), mk(2, 1, 4, 101, (1, 0)), mk(2, 2, 12, 13, (1, 2))]
    for i, d in enumerate(cases):
        check(d, 3300 + i)
        check(d, 3400 + i, ties=True)
