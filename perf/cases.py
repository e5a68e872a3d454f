"""The work users have this library do, as cases that can be timed and compared.

A case is one pass through the public layers (`paper_2504_06881_b200.nn`) on device tensors:
inference (`direction` "infer": the forward under `torch.no_grad`) or one training pass ("train":
forward, then every gradient through autograd).  `kind` names the layer class: "2d" TropicalConv2d,
"dw" TropicalDepthwiseConv2d, "1d" TropicalConv1d, "3d" TropicalConv3d.  Sizes are those of the
library's benchmark configurations (`inputs.py`, `bench.py`) and of the networks the paper trains.
"""
import math

import torch

from paper_2504_06881_b200 import nn as tnn


def _case(name, kind, direction, mode, dtype, N, C, K, size, k, stride=1, dil=1, x="f32", grad_x=True,
          chan="default", bias=True, relu=False, wstd=0.1, pad=None):
    D, H, W = (1,) * (3 - len(size)) + tuple(size)
    c = dict(kind=kind, direction=direction, mode=mode, chan=chan, dtype=dtype, x=x, N=N, C=C, K=K, D=D, H=H, W=W,
             k=k, stride=stride, dil=dil, pad=dil * (k - 1) // 2 if pad is None else pad, grad_x=grad_x, bias=bias,
             relu=relu, wstd=wstd)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one image through the opening layer of LeNet: the latency of the smallest call
        _case("lenet_open_infer", "2d", "infer", "compound", "f32", 1, 1, 6, (28, 28), 5),
        # the small configuration of the benchmark set: two RGB images, 3 -> 16 channels
        _case("small_rgb_train", "2d", "train", "compound", "f32", 2, 3, 16, (32, 32), 3, wstd=0.3),
        # CIFAR-sized hidden layer, a full training batch: the max-plus layer and the compound layer
        _case("cifar_maxplus_train", "2d", "train", "max_plus", "f32", 128, 64, 64, (32, 32), 3),
        _case("cifar_compound_train", "2d", "train", "compound", "f32", 128, 64, 64, (32, 32), 3),
        # ImageNet-scale middle layers, a parallel network: the stride-2 transition in fp32, a 28x28 layer in bf16
        _case("imagenet_s2_parallel_train", "2d", "train", "parallel", "f32", 64, 64, 128, (56, 56), 3, stride=2,
              bias=False, wstd=0.05),
        _case("imagenet_28_parallel_bf16_train", "2d", "train", "parallel", "bf16", 64, 128, 128, (28, 28), 3,
              x="bf16", bias=False, wstd=0.05),
        # last stage of the hybrid ResNet-18: fp32 activations around a bf16 layer, 7x7 maps
        _case("resnet_last_compound_bf16_train", "2d", "train", "compound", "bf16", 64, 512, 512, (7, 7), 3,
              bias=False, wstd=0.05),
        # segmentation-scale feature map with atrous windows: the largest training pass
        _case("segmentation_compound_bf16_train", "2d", "train", "compound", "bf16", 8, 256, 256, (128, 256), 3,
              dil=2, x="bf16", relu=True, wstd=0.05),
        # a served classifier's middle layer, a modest batch
        _case("imagenet_28_compound_infer", "2d", "infer", "compound", "f32", 16, 128, 128, (28, 28), 3, wstd=0.05),
        # MobileNetV2's expanded 24-channel stage: depthwise layer in training
        _case("mobilenet_depthwise_train", "dw", "train", "compound", "f32", 128, 144, 144, (56, 56), 3),
        # opening layer of an audio network: 80 samples at stride 4 on raw signals, no gradient for the input
        _case("audio_open_train", "1d", "train", "compound", "f32", 32, 1, 128, (16000,), 80, stride=4, pad=0,
              grad_x=False),
        # second layer of the 3-D LeNet on 28^3 volumes
        _case("lenet3d_train", "3d", "train", "compound", "f32", 32, 6, 16, (6, 6, 6), 5, pad=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: odd and ragged sizes among them, no dearer than the largest listed."""
    kind = rng.choices(["2d", "dw", "1d", "3d"], [6, 1.5, 1, 1])[0]
    direction = rng.choices(["train", "infer"], [7, 3])[0]
    mode = rng.choices(["max_plus", "min_plus", "compound", "parallel"], [1.5, 1, 3, 2])[0]
    dtype = rng.choice(["f32", "bf16"])
    x = "f32" if dtype == "f32" else rng.choice(["f32", "bf16"])
    chan = "default"
    bias, relu = rng.random() < 0.5, rng.random() < 0.3
    N = _log_int(rng, 1, 128)
    stride, dil, grad_x, pad = 1, 1, True, None
    if kind == "2d":
        if mode in ("max_plus", "min_plus"):
            chan = rng.choice(["default", "default", "sum"])
        k = rng.choice([3, 3, 3, 3, 5])
        if k == 3:
            stride, dil = rng.choice([(1, 1), (1, 1), (1, 1), (2, 1), (1, 2), (1, 4)])
        C, K = _log_int(rng, 1, 512), _log_int(rng, 4, 512)
        H = _log_int(rng, 7, 128)
        size = (H, min(256, max(7, int(H * rng.uniform(0.7, 2.0)))))
        # at most 2e10 taps (a seventh of the largest listed case)
        N = max(1, min(N, int(2e10 / (C * K * k * k * size[0] * size[1] / stride ** 2))))
        while N == 1 and C * K * k * k * size[0] * size[1] / stride ** 2 > 2e10:
            C, K = max(1, C * 2 // 3), max(4, K * 2 // 3)
        grad_x = C > 3
    elif kind == "dw":
        k, stride = 3, rng.choice([1, 1, 2])
        C = K = _log_int(rng, 16, 576)
        H = _log_int(rng, 7, 112)
        size = (H, H)
        N = max(1, min(N, int(8e7 / (C * H * H))))
    elif kind == "1d":
        k, stride = rng.choice([(3, 1), (3, 1), (80, 4), (80, 4), (9, 1), (21, 2)])
        C = 1 if k == 80 else _log_int(rng, 1, 64)
        K = _log_int(rng, 8, 128)
        L = _log_int(rng, 250, 16000)
        size, pad = (L,), 0 if k == 80 else k // 2
        N = max(1, min(N, 64, int(2e9 / (C * K * k * L / stride))))
        grad_x = C > 1
    else:
        k = rng.choice([3, 5])
        stride = rng.choice([1, 2])
        C, K = _log_int(rng, 1, 16), _log_int(rng, 6, 32)
        E = _log_int(rng, 6, 48)
        size, pad = (E, E, E), rng.choice([0, k // 2])
        N = max(1, min(N, 32, int(1e9 / (C * K * k ** 3 * E ** 3 / stride ** 3))))
        grad_x = C > 1
    return _case(None, kind, direction, mode, dtype, N, C, K, size, k, stride, dil, x, grad_x, chan, bias, relu,
                 0.1, pad)


_X_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


def _spatial(c):
    return {"1d": (c["W"],), "2d": (c["H"], c["W"]), "dw": (c["H"], c["W"]), "3d": (c["D"], c["H"], c["W"])}[c["kind"]]


def _out(c):
    return tuple((s + 2 * c["pad"] - c["dil"] * (c["k"] - 1) - 1) // c["stride"] + 1 for s in _spatial(c))


def prepare(case, seed):
    """A layer with trained-looking weights, a batch of normalised activations and an upstream gradient."""
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    randn = lambda *s: torch.randn(*s, device="cuda", generator=gen)
    args = dict(stride=c["stride"], padding=c["pad"], dilation=c["dil"], bias=c["bias"], mode=c["mode"], dtype=c["dtype"])
    if c["kind"] == "dw":
        layer = tnn.TropicalDepthwiseConv2d(c["C"], c["k"], **args)
    else:
        cls = {"1d": tnn.TropicalConv1d, "2d": tnn.TropicalConv2d, "3d": tnn.TropicalConv3d}[c["kind"]]
        layer = cls(c["C"], c["K"], c["k"], chan=c["chan"], **args)
    layer = layer.cuda()
    with torch.no_grad():
        for name, p in layer.named_parameters():
            last = name.rsplit(".", 1)[-1]
            if last in ("alpha", "beta"):
                p.copy_(torch.rand(p.shape, device="cuda", generator=gen))
            elif last == "bias":
                p.copy_(torch.rand(p.shape, device="cuda", generator=gen) * 0.2 - 0.1)
            else:
                p.copy_(randn(*p.shape) * c["wstd"])
    x = randn(c["N"], c["C"], *_spatial(c))
    if c["relu"]:
        x = x.relu_()
    x = x.to(_X_DTYPE[c["x"]])
    state = {"layer": layer, "x": x, "train": c["direction"] == "train"}
    if state["train"]:
        x.requires_grad_(c["grad_x"])
        state["wanted"] = ([x] if c["grad_x"] else []) + list(layer.parameters())
        state["g"] = randn(c["N"], c["K"], *_out(c)).to(x.dtype)
    return state


def run(state):
    """Inference: the layer's output.  Training: the output and the gradients of input and parameters."""
    if not state["train"]:
        with torch.no_grad():
            return state["layer"](state["x"])
    y = state["layer"](state["x"])
    return (y.detach(),) + torch.autograd.grad(y, state["wanted"], state["g"])


def work(case):
    """Bytes: each input read once, each output written once.  Operations: one add and one compare per
    tap and branch (compound shares the add), two multiplications and two sums per branch and channel;
    backward: per routed winner one accumulation into grad_x and one into grad_w, scaled where the layer
    has alpha / beta, and a multiply-add for each of their gradients."""
    c = case
    es = 4 if c["x"] == "f32" else 2
    taps = c["k"] ** len(_spatial(c))
    two, dw = c["mode"] in ("compound", "parallel"), c["kind"] == "dw"
    cin = 1 if dw else c["C"]
    nx = c["N"] * c["C"] * math.prod(_spatial(c))
    ny = c["N"] * c["K"] * math.prod(_out(c))
    nw = c["K"] * cin * taps * (2 if c["mode"] == "parallel" else 1) + (2 * c["K"] * cin if two else 0) + c["K"] * c["bias"]
    pairs = ny * cin                                  # (output, input channel)
    per_tap = {"compound": 3, "parallel": 4}.get(c["mode"], 2)
    nbytes, ops = (nx + ny) * es + nw * 4, pairs * (taps * per_tap + (4 if two else 1))
    if c["direction"] == "train":
        nbytes += (ny + (nx if c["grad_x"] else 0)) * es + nw * 4
        summed = two or c["chan"] == "sum" or dw
        routed = (pairs if summed else ny) * (2 if two else 1)
        ops += routed * ((2 if two else 1) * c["grad_x"] + 1 + (2 if two else 0))
    return {"bytes": nbytes, "flops": ops}


def tolerance(case):
    """fp32 layers differ by the order of their fp32 sums only; bf16 layers round outputs to 8 bits."""
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}
