"""Layers called without gradient recording run the winner-free kernels and give the same outputs."""
import pytest
import torch

from paper_2504_06881_b200 import nn as tnn, tconv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("no_grad", [torch.no_grad, torch.inference_mode])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["max_plus", "compound"])
def test_no_winners_without_recording(mode, dtype, no_grad):
    torch.manual_seed(5)
    layer = tnn.TropicalConv2d(5, 9, 3, padding=1, mode=mode, dtype=dtype).cuda()
    x = torch.randn(2, 5, 12, 16, device="cuda")
    y = layer(x)
    assert y.requires_grad and "win" in tconv.tconv_last_kernel()
    with no_grad():
        z = layer(x)
    assert not z.requires_grad and "win" not in tconv.tconv_last_kernel()
    assert torch.equal(y.detach(), z)
