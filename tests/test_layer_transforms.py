"""The layers under the tools of torch.autograd: saved-tensor hooks, recomputation, forward-mode differentiation,
tracing and the function transforms.  What the native path cannot serve has to be refused or to take another path."""
import pytest
import torch
import torch.autograd.forward_ad as fwad
from torch.utils.checkpoint import checkpoint

from paper_2504_06881_b200 import nn as tnn

KINDS = {
    "dense": (lambda **kw: tnn.TropicalConv2d(4, 5, 3, padding=1, **kw), (2, 4, 9, 10)),
    "dense_max": (lambda **kw: tnn.TropicalConv2d(4, 5, 3, padding=1, mode="max_plus", **kw), (2, 4, 9, 10)),
    "depthwise": (lambda **kw: tnn.TropicalDepthwiseConv2d(4, 3, padding=1, **kw), (2, 4, 9, 10)),
    "volume": (lambda **kw: tnn.TropicalConv3d(4, 5, 3, padding=1, **kw), (2, 4, 5, 6, 7)),
    "signal": (lambda **kw: tnn.TropicalConv1d(4, 5, 7, **kw), (2, 4, 30)),
}


def make(kind, device="cuda", **kw):
    torch.manual_seed(3)
    layer, shape = KINDS[kind]
    return layer(**kw).to(device), torch.randn(shape, device=device)


def gradients(m, x, call=None):
    x = x.clone().requires_grad_()
    y = (call or m)(x)
    return torch.autograd.grad(y, [x] + list(m.parameters()), torch.ones_like(y))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("kind", KINDS)
def test_saved_tensors_elsewhere(kind, dtype):
    m, x = make(kind, dtype=dtype)
    ref = gradients(m, x)
    with torch.autograd.graph.save_on_cpu():
        got = gradients(m, x)
    assert all(torch.equal(a, b) for a, b in zip(ref, got))
    got = gradients(m, x, lambda v: checkpoint(m, v, use_reentrant=False))
    assert all(torch.equal(a, b) for a, b in zip(ref, got))


@pytest.mark.gpu
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("pack", [
    lambda t: t.cpu(),                                                   # not brought back
    lambda t: t.half() if t.is_floating_point() else t,                  # another type
    lambda t: t.int() if not t.is_floating_point() else t,
    lambda t: t.flatten()[: t.numel() // 2],                             # another size
    lambda t: t.repeat_interleave(2, -1)[..., ::2],                      # strided
], ids=["host", "half", "int", "short", "strided"])
def test_other_saved_tensors_are_refused(kind, pack):
    m, x = make(kind)
    x.requires_grad_()
    with torch.autograd.graph.saved_tensors_hooks(pack, lambda t: t):
        y = m(x)
    with pytest.raises(ValueError):
        y.sum().backward()


@pytest.mark.parametrize("kind", ["dense", "depthwise", "volume"])
@pytest.mark.parametrize("record", [True, False])
def test_forward_mode_is_refused(kind, record):
    m, x = make(kind, "cpu")
    with torch.set_grad_enabled(record), fwad.dual_level(), pytest.raises(NotImplementedError):
        m(fwad.make_dual(x, torch.ones_like(x)))


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["dense", "depthwise", "volume"])
def test_geometry_as_lists(kind):
    m, x = make(kind)
    ref = m(x)
    m.stride, m.padding, m.dilation = list(m.stride), list(m.padding), list(m.dilation)
    assert torch.equal(m(x), ref)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("record", [True, False])
def test_traced_layers_compute(kind, record):
    m, x = make(kind)
    for p in m.parameters():
        p.requires_grad_(record)
    traced = torch.jit.trace(m, x, check_trace=False)
    other = torch.randn_like(x)
    assert torch.equal(traced(other), m(other))
    if record:
        assert all(torch.equal(a, b) for a, b in zip(gradients(m, other), gradients(m, other, traced)))


@pytest.mark.gpu
@pytest.mark.parametrize("kind", KINDS)
def test_transforms_are_refused(kind):
    m, x = make(kind)
    with pytest.raises(RuntimeError):
        torch.func.vmap(m)(torch.stack([x, x]))
    with pytest.raises(RuntimeError), torch.no_grad():
        torch.func.vmap(m)(torch.stack([x, x]))
    with pytest.raises(RuntimeError):
        torch.func.grad(lambda v: m(v).sum())(x)


@pytest.mark.gpu
def test_functions_take_the_geometry_alone():
    m, x = make("dense")
    geom = (m.mode, m.chan, m.dtype, m.stride, m.padding, m.dilation)
    y = tnn.TropicalConvFn.apply(x, m.weight, m.weight2, m.alpha, m.beta, m.bias, geom)
    assert torch.equal(y, m(x)) and y.requires_grad
