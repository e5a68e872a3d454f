"""Host-side plans of the backward kernels: no other count of chunks has less work in its rounds of resident blocks."""
import pytest

from paper_2504_06881_b200 import inputs, tconv

ceil = lambda a, b: -(-a // b)


def dw_chunks(d):
    OH, OW = inputs.output_hw(d)
    codes = ceil(d["N"] * d["C"] * OH * OW, 256) * 256
    return (tconv.tconv_dw_workspace_bytes(d, True) - codes - 256) // (d["C"] * 35 * 4)


def dw_cost(d, chunks):
    """Rounds of resident blocks times half-steps (of a warp's strips, of 1024 outputs), for the kernel that runs."""
    N, C = d["N"], d["C"]
    OH, OW = inputs.output_hw(d)
    items = N * OH * OW
    strips = d["R"] == d["S"] == 3 and d["dil_w"] == 1 and d["stride_w"] <= 2 and OH * OW >= 100 and \
        min(ceil(592, C), ceil(items, 1024)) <= 2 * N
    if not strips:
        return ceil(C * chunks, 592) * (2 * ceil(ceil(items, chunks), 1024) + 4)
    vec = d["pad_w"] == 1 and d["W"] % 4 == 0
    two = d["mode"] == "parallel" and d["stride_w"] == 2 and not (d["dtype"] == "bf16" and vec)
    return ceil(C * chunks, 148 * (2 if two else 3)) * (2 * ceil(ceil(N, chunks) * ceil(OW, 4) * ceil(OH, 6), 32) + 16)


SHAPES = [(128, 84, 7, 1, 1), (128, 148, 7, 1, 1), (64, 160, 7, 1, 1), (64, 320, 7, 1, 1), (64, 148, 28, 1, 2), (64, 296, 28, 1, 2),
          (64, 144, 56, 1, 1), (128, 144, 56, 1, 1), (64, 144, 56, 2, 1), (64, 144, 57, 1, 1), (32, 576, 14, 1, 1), (128, 16, 28, 1, 1),
          (16, 384, 14, 1, 1), (13, 66, 21, 2, 1), (2, 64, 56, 1, 1), (1, 32, 224, 1, 1), (4, 144, 56, 1, 1), (128, 1, 28, 1, 1),
          (100, 720, 7, 2, 1), (1, 1, 5, 1, 1), (31, 37, 61, 1, 1)]


@pytest.mark.parametrize("mode,dtype", [("compound", "f32"), ("parallel", "f32"), ("parallel", "bf16"), ("max_plus", "bf16")])
def test_depthwise_chunks(mode, dtype):
    for N, C, E, s, dil in SHAPES:
        d = inputs.layer(N, C, E, E, C, stride=s, pad=dil, dil=dil, mode=mode, dtype=dtype)
        OH, OW = inputs.output_hw(d)
        most = N if OH * OW >= 100 and dil == 1 else ceil(N * OH * OW, 1024)
        got = dw_chunks(d)
        assert 1 <= got <= N * OH * OW
        best = min(dw_cost(d, c) for c in range(1, min(most, 4 * ceil(592, C)) + 1))
        assert dw_cost(d, got) <= best, (d, got, dw_cost(d, got), best)
