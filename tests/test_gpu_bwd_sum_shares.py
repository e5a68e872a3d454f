"""Parameter gradients of the Sum forms where the loops over a share's items and over the partial rows change: images of one
and of several whole blocks of 128 quads, rounds that are not whole blocks, flattened ranges around the eight rounds of a step
and their last partial round, shares of one block, one or two branches and wide codes; slices of no row to seventeen."""
import pytest

from nvcc_probe import sum_gw_plans
from paper_2504_06881_b200 import inputs, tconv
import parity

pytestmark = pytest.mark.gpu

L = inputs.layer
LAYERS = [
    L(1, 1, 16, 32, 1, pad=1),                           # one block
    L(3, 2, 16, 32, 3, pad=1),                           # three images of one block, an odd number of blocks
    L(9, 3, 32, 32, 4, pad=1),                           # two blocks an image, several shares
    L(5, 2, 16, 24, 3, pad=1),                           # three rounds an image: whole rounds, no blocks
    L(2, 2, 32, 48, 3, pad=1),                           # three blocks an image
    L(1, 2, 11, 23, 3, pad=1),                           # flattened: 66 quads
    L(4, 3, 24, 16, 5, pad=0),                           # flattened: 88 quads an image, 11 rounds
    L(7, 2, 13, 61, 4, pad=1),                           # flattened: 208 quads an image, 45 rounds and a last one of 16 lanes
    L(32, 1, 20, 20, 2, pad=1),                          # flattened: 100 rounds, a last one of 4 lanes
    L(3, 2, 16, 32, 3, R=5, S=5, pad=2),                 # wide codes, one block
    L(3, 2, 9, 21, 3, R=5, S=5, pad=2),                  # wide codes, flattened
]


@pytest.mark.parametrize("mode", ["compound", "parallel", "max_plus"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_shares(mode, dtype):
    for i, d in enumerate(LAYERS):
        parity.check_layer(dict(d, mode=mode, chan="sum", dtype=dtype), None, 2700 + i, recompute=False)
        assert tconv.tconv_last_kernel() == "bwd_sum", d


@pytest.mark.parametrize("N", [1, 4, 5, 30, 32, 33, 129, 144, 161, 272])
def test_partial_rows(N):
    """4, 16, 20, 120, 128, 132 rows of grad_alpha / grad_beta (four tiles an image), then one an image, in sixteen slices."""
    parity.check_layer(dict(L(N, 2, 16, 64, 5, pad=1), mode="compound", chan="sum", dtype="f32"), None, 2800 + N, recompute=False)
    assert tconv.tconv_last_kernel() == "bwd_sum"


@pytest.mark.parametrize("mode", ["max_plus", "min_plus"])
def test_one_round_of_eight(mode):
    """fp32, one branch, wide codes: more CTAs than seven per SM, with shares of 52 rounds (whole blocks) and of 64 (whole rounds)."""
    layers = [L(50, 13, 16, 96, 29, R=5, S=5, pad=2), L(32, 24, 32, 64, 24, R=5, S=5, pad=2)]
    for i, (d, per) in enumerate(zip(layers, (52, 64))):
        d = dict(d, mode=mode, chan="sum", dtype="f32")
        plan, = sum_gw_plans([d])
        assert plan["blocks"] and plan["per"] == per and 148 * 28 < d["C"] * d["K"] * plan["splits"] <= 148 * 32
        parity.check_layer(d, None, 2900 + i, recompute=False)
        assert tconv.tconv_last_kernel() == "bwd_sum"


@pytest.mark.parametrize("mode,layer", [("compound", L(40, 3, 11, 23, 4, pad=1)), ("parallel", L(9, 3, 31, 37, 4, pad=1)),
                                        ("max_plus", L(17, 3, 13, 61, 4, pad=1)), ("compound", L(17, 3, 13, 61, 4, R=5, S=5, pad=2)),
                                        ("min_plus", L(64, 3, 11, 23, 4, R=5, S=5, pad=2))])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_flattened_shares(mode, layer, dtype):
    """Several shares of more than twelve rounds that start and end inside an image; the last one shorter in three layers."""
    d = dict(layer, mode=mode, chan="sum", dtype=dtype)
    OH, OW = inputs.output_hw(d)
    quads = OH * ((OW + 3) // 4)
    plan, = sum_gw_plans([d])
    assert plan["flat"] and plan["splits"] >= 6 and plan["per"] > 12 * 32 and plan["per"] % quads and plan["per"] % 32
    parity.check_layer(d, None, 2950, recompute=False)
    assert tconv.tconv_last_kernel() == "bwd_sum"
