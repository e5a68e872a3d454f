"""Parameter gradients of 3x3 depthwise layers where their strips and chunks change: planes of one row of strips with a
short last row, widths that are not whole quads, equal winners in neighbouring outputs (ties everywhere), one chunk and
several, images or outputs that the chunks do not divide, planes of the strips and of the any-window kernel, strides 1 and
2, both types."""
import pytest

from paper_2504_06881_b200 import inputs
from test_backward_plans import dw_chunks
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


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["compound", "parallel", "min_plus"])
def test_uneven_chunks(mode, dtype):
    mk = lambda N, C, H, W, s=1, d=1: inputs.layer(N, C, H, W, C, 3, 3, mode=mode, dtype=dtype, stride=s, pad=d, dil=d)
    cases = [(mk(13, 150, 20, 20), 2), (mk(11, 37, 29, 28), 11), (mk(6, 64, 30, 30), 6),
             (mk(11, 100, 24, 25, 2), 2 if mode == "parallel" else 3),                        # strips
             (mk(63, 160, 7, 7), 2), (mk(50, 31, 7, 9), 4), (mk(13, 296, 28, 28, 1, 2), 2)]      # any window
    for i, (d, chunks) in enumerate(cases):
        assert dw_chunks(d) == chunks, d
        check(d, 3700 + i)
