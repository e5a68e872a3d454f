"""The layers' native autograd path: the same bits as the binding's forward / backward for every combination of
optional tensors, None gradients where none is wanted, and the binding's errors."""
import pytest
import torch

from paper_2504_06881_b200 import nn as tnn, tconv, tconv3d

pytestmark = pytest.mark.gpu

KW = dict(mode=["max_plus", "compound", "parallel"], params=["2p", "0p"], bias=[True, False], dtype=["f32", "bf16"])


@pytest.mark.parametrize("dtype", KW["dtype"])
@pytest.mark.parametrize("bias", KW["bias"])
@pytest.mark.parametrize("params", KW["params"])
@pytest.mark.parametrize("mode", KW["mode"])
@pytest.mark.parametrize("kind", ["dense", "depthwise", "volume"])
def test_same_as_the_binding(kind, mode, params, bias, dtype):
    torch.manual_seed(7)
    args = dict(padding=1, mode=mode, params=params, bias=bias, dtype=dtype)
    dt = tconv.TORCH_DTYPE[dtype]
    if kind == "depthwise":
        m, shape, fwd, bwd = tnn.TropicalDepthwiseConv2d(6, 3, **args), (2, 6, 9, 10), tconv.dw_forward, tconv.dw_backward
        d = dict(N=2, C=6, H=9, W=10, K=6, R=3, S=3, stride_h=1, stride_w=1, pad_h=1, pad_w=1, dil_h=1, dil_w=1, chan="sum")
    elif kind == "dense":
        m, shape, fwd, bwd = tnn.TropicalConv2d(4, 5, 3, **args), (2, 4, 9, 10), tconv.forward, tconv.backward
        d = dict(N=2, C=4, H=9, W=10, K=5, R=3, S=3, stride_h=1, stride_w=1, pad_h=1, pad_w=1, dil_h=1, dil_w=1, chan="default")
    else:
        m, shape, fwd, bwd = tnn.TropicalConv3d(4, 5, 3, **args), (2, 4, 5, 6, 7), tconv3d.forward, tconv3d.backward
        d = dict(N=2, C=4, D=5, H=6, W=7, K=5, T=3, R=3, S=3, stride=(1, 1, 1), pad=(1, 1, 1), dil=(1, 1, 1), chan="default")
    d.update(mode=mode, dtype=dtype)
    m = m.cuda()
    x = torch.randn(shape, device="cuda", requires_grad=True)
    y = m(x)
    g = torch.randn_like(y)
    names = [n for n, _ in m.named_parameters()]
    got = dict(zip(["x"] + names, torch.autograd.grad(y, [x] + list(m.parameters()), g)))
    c = lambda t: None if t is None else t.detach().to(dt)
    f = lambda t: None if t is None else t.detach()
    y1, win = fwd(d, c(x), c(m.weight), c(m.weight2), f(m.alpha), f(m.beta), f(m.bias), want_winners=True)
    assert torch.equal(y, y1.float())
    ref = bwd(d, c(x), c(m.weight), c(g), c(m.weight2), f(m.alpha), f(m.beta), win)
    keys = dict(x="grad_x", weight="grad_w", weight2="grad_w2", alpha="grad_alpha", beta="grad_beta", bias="grad_bias")
    for n, v in got.items():
        assert torch.equal(v, ref[keys[n]].float()), n
    y = m(x.detach())                      # an input that needs no gradient: its kernel is skipped, the rest is the same
    for n, v in zip(names, torch.autograd.grad(y, list(m.parameters()), g)):
        assert torch.equal(v, got[n]), n


def test_errors():
    m = tnn.TropicalConv2d(4, 5, 3).cuda()
    with pytest.raises(ValueError):
        m(torch.randn(1, 4, 8, 8))                        # host tensor
    with pytest.raises(ValueError):
        m(torch.randn(1, 3, 8, 8, device="cuda"))         # other channel count
    with pytest.raises(ValueError):
        m(torch.randn(4, 8, 8, device="cuda"))
    with pytest.raises(tconv.TconvError):
        m(torch.randn(1, 4, 2, 8, device="cuda"))         # window larger than the input
