"""Parameter gradients of 3x3 depthwise layers where their strips and chunks change: planes of one row of strips with a
short last row, widths that are not whole quads, equal winners in neighbouring outputs (ties everywhere), one chunk and
several, strides 1 and 2, both types."""
import pytest

from paper_2504_06881_b200 import inputs
from test_gpu_depthwise import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["compound", "parallel", "max_plus", "min_plus"])
def test_strips_and_chunks(mode, dtype):
    mk = lambda N, C, H, W, s: inputs.layer(N, C, H, W, C, 3, 3, mode=mode, dtype=dtype, stride=s, pad=1)
    cases = [mk(1, 2, 6, 20, 1), mk(2, 2, 7, 17, 1), mk(2, 3, 25, 10, 2), mk(3, 1, 26, 23, 2), mk(12, 160, 12, 13, 1),
             mk(12, 150, 23, 24, 2)]
    for i, d in enumerate(cases):
        check(d, 3500 + i)
        check(d, 3600 + i, ties=True)
