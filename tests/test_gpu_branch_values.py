"""grad_alpha / grad_beta are sums of grad_y times the branch values as the forward rounded them.  Tolerance: the
products of the bf16 layers are exact in fp32 and a value passes fewer than 100 fp32 additions, so that the result
is within 100 * 2^-24 < 1e-5 of the sum of |contributions|; fp32 layers round each branch value and product as well.
Also: what cancels inside a branch value does not reach the sums, and taps that never win add nothing, whatever
their weight (infinite weights are how a caller masks a tap: +inf under min, -inf under max)."""
import numpy as np
import pytest
import torch

from oracle import tconv3d_oracle as ora3, tconv_oracle as ora
from paper_2504_06881_b200 import inputs, tconv, tconv3d
import parity

pytestmark = pytest.mark.gpu

L = inputs.layer
RTOL = 1e-5
PARAMS = ("grad_w", "grad_w2", "grad_alpha", "grad_beta", "grad_bias")
LAYERS = [
    L(2, 3, 32, 32, 33, pad=1),                     # one tile of 256 quads, output channels past a whole stage
    L(1, 2, 37, 70, 9, pad=2, dil=2),               # several tiles, ragged rows
    L(19, 3, 7, 7, 12, stride=2, pad=1),            # several images per tile
    L(2, 2, 20, 23, 5, R=5, S=5, pad=2),            # 16-bit codes
    L(1, 2, 24, 25, 3, R=4, S=4, pad=1),
]


def device_grads(d, t, winners=None):
    g = parity.to_dev(t, d)
    la = parity.layer_args(d, g)
    if winners is None:
        _, winners = tconv.forward(d, g["x"], g["w"], la["w2"], la["alpha"], la["beta"], g["bias"], want_winners=True)
    return tconv.backward(d, g["x"], g["w"], g["g"], la["w2"], la["alpha"], la["beta"], winners)


def oracle_grads(d, t):
    la = parity.layer_args(d, t)
    return ora.backward(d, t["x"], t["w"], t["g"], la["w2"], la["alpha"], la["beta"])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["compound", "parallel"])
def test_dense(mode, dtype):
    for i, d in enumerate(LAYERS):
        d = dict(d, mode=mode, dtype=dtype)
        t = inputs.draw(d, 4100 + i)
        got, ref = device_grads(d, t), oracle_grads(d, t)
        assert tconv.tconv_last_kernel() == "bwd_sum"
        parity.compare_grads(d, {k: got[k] for k in PARAMS if k in got}, ref, rtol=RTOL)


@pytest.mark.parametrize("mode", ["compound", "parallel"])
def test_dense_offset_inputs(mode):
    """Inputs around 4096 under weights around -4096: |x| and |w| are thousands of times |x + w|."""
    for i, d in enumerate(LAYERS[:3]):
        d = dict(d, mode=mode, dtype="f32", pad_h=0, pad_w=0)
        t = inputs.draw(d, 4200 + i, x=("normal", 4096.0, 1.0), w=("normal", -4096.0, 1.0))
        parity.compare_grads(d, device_grads(d, t), oracle_grads(d, t), rtol=RTOL)


def masked(t):
    """Every other tap of the min branch and the others of the max branch masked (the middle one in neither)."""
    taps = t["w"].reshape(t["w"].shape[:2] + (-1,)).shape[2]
    keep = taps // 2
    for name, start, v in (("w", 0, np.inf), ("w2", 1, -np.inf)):
        flat = t[name].reshape(t[name].shape[:2] + (taps,))
        flat[..., [i for i in range(start, taps, 2) if i != keep]] = v
    return t


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_dense_masked_taps(dtype):
    for i, d in enumerate(LAYERS[:3]):
        d = dict(d, mode="parallel", dtype=dtype)
        t = masked(inputs.draw(d, 4300 + i))
        ref = ora.forward(d, t["x"], t["w"], t["w2"], t["alpha"], t["beta"], t["bias"])
        # (the fp32 forward recovers winners from differences of tap sums, which infinite sums do not have: the
        # oracle's winners are passed to the backward)
        OH, OW = inputs.output_hw(d)
        codes = np.zeros((d["N"], d["K"], d["C"], OH, (OW + 3) // 4 * 4), np.uint8)
        codes[..., :OW] = ref["codes"]
        got = device_grads(d, t, torch.from_numpy(codes).cuda().reshape(-1))
        parity.compare_grads(d, {k: got[k] for k in PARAMS}, oracle_grads(d, t), rtol=RTOL)


@pytest.mark.parametrize("mode,chan", [("compound", "sum"), ("parallel", "sum"), ("max_plus", "sum")])
@pytest.mark.parametrize("K", [8, 9, 12])
def test_dense_infinite_gradient(mode, chan, K):
    """One infinite gradient in the last output channel reaches its winners' inputs as an infinity, nothing else."""
    for i, shape in enumerate([dict(N=2, C=3, H=12, W=13), dict(N=1, C=2, H=40, W=72)]):
        d = L(shape["N"], shape["C"], shape["H"], shape["W"], K, pad=1, mode=mode, chan=chan)
        t = inputs.draw(d, 4400 + i)
        t["alpha"] += 0.5
        t["beta"] += 0.5
        t["g"][0, K - 1, 5, 6] = np.inf
        got = device_grads(d, t)["grad_x"].cpu().numpy()
        ref = oracle_grads(d, t)["grad_x"][0]
        assert not np.isnan(got).any()
        assert np.array_equal(np.isinf(got), np.isinf(ref)) and np.isinf(got).any()


VOLUMES = [
    inputs.layer3d(4, 6, 6, 6, 6, 16, T=5, R=5, S=5),
    inputs.layer3d(2, 3, 9, 11, 10, 8, T=3, R=3, S=3, stride=(2, 3, 2), pad=1, dil=(1, 2, 1)),
    inputs.layer3d(3, 2, 1, 9, 40, 3, T=1, R=3, S=3, pad=(0, 1, 1)),
]


def volume_grads(d, t):
    dt = tconv.TORCH_DTYPE[d["dtype"]]
    dev = {k: torch.from_numpy(v).cuda().to(dt if k in ("x", "w", "w2", "g") else torch.float32) for k, v in t.items()}
    w2 = dev["w2"] if d["mode"] == "parallel" else None
    _, win = tconv3d.forward(d, dev["x"], dev["w"], w2, dev["alpha"], dev["beta"], dev["bias"], want_winners=True)
    return tconv3d.backward(d, dev["x"], dev["w"], dev["g"], w2, dev["alpha"], dev["beta"], win)


def check_volume(d, t):
    got = volume_grads(d, t)
    ref = ora3.backward(d, t["x"], t["w"], t["g"], t["w2"] if d["mode"] == "parallel" else None, t["alpha"], t["beta"])
    parity.compare_grads(d, {k: got[k] for k in PARAMS if k in got}, ref, rtol=RTOL)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["compound", "parallel"])
def test_volume(mode, dtype):
    for i, d in enumerate(VOLUMES):
        d = dict(d, mode=mode, dtype=dtype)
        check_volume(d, inputs.draw3d(d, 4500 + i))


@pytest.mark.parametrize("mode", ["compound", "parallel"])
def test_volume_offset_inputs(mode):
    for i, d in enumerate(VOLUMES):
        d = dict(d, mode=mode, pad=(0, 0, 0))
        check_volume(d, inputs.draw3d(d, 4600 + i, x=("normal", 4096.0, 1.0), w=("normal", -4096.0, 1.0)))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_volume_masked_taps(dtype):
    for i, d in enumerate(VOLUMES):
        d = dict(d, mode="parallel", dtype=dtype)
        check_volume(d, masked(inputs.draw3d(d, 4700 + i)))


def depthwise(d, t):
    """Gradients of a depthwise layer and the oracle's."""
    dt, par = tconv.TORCH_DTYPE[d["dtype"]], d["mode"] == "parallel"
    dev = {k: torch.from_numpy(v).cuda().to(dt if k in ("x", "w", "w2", "g") else torch.float32) for k, v in t.items()}
    w2 = dev["w2"] if par else None
    _, win = tconv.dw_forward(d, dev["x"], dev["w"], w2, dev["alpha"], dev["beta"], None, want_winners=True)
    got = tconv.dw_backward(d, dev["x"], dev["w"], dev["g"], w2, dev["alpha"], dev["beta"], win)
    return got, ora.depthwise_backward(d, t["x"], t["w"], t["g"], t["w2"] if par else None, t["alpha"], t["beta"])


DEPTHWISE = [L(3, 4, 12, 12, 4, pad=1), L(2, 3, 37, 9, 3, pad=1), L(5, 2, 33, 46, 2, pad=(2, 1)), L(3, 2, 14, 13, 2, stride=2)]


def draw_depthwise(d, seed, x=("normal", 0.0, 1.0), w=("normal", 0.0, 0.3)):
    t = inputs.draw(dict(d, C=1, K=d["C"]), seed, x=x, w=w)          # weights [C][1][R][S], one alpha and beta per channel
    t["x"], t["g"] = (inputs.draw(dict(d, K=d["C"]), seed, x=x)[k] for k in ("x", "g"))
    t["w"], t["w2"] = (np.ascontiguousarray(t[k][:, 0]) for k in ("w", "w2"))
    t["alpha"], t["beta"] = (np.ascontiguousarray(t[k][:, 0]) for k in ("alpha", "beta"))
    return t


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["compound", "parallel"])
def test_depthwise(mode, dtype):
    for i, d in enumerate(DEPTHWISE):
        d = dict(d, mode=mode, dtype=dtype)
        got, ref = depthwise(d, draw_depthwise(d, 4800 + i))
        parity.compare_grads(d, {k: got[k] for k in PARAMS if k in got}, ref, rtol=RTOL)


@pytest.mark.parametrize("mode", ["compound", "parallel"])
def test_depthwise_offset_inputs(mode):
    for i, d in enumerate(DEPTHWISE):
        d = dict(d, mode=mode, pad_h=0, pad_w=0)
        got, ref = depthwise(d, draw_depthwise(d, 4900 + i, x=("normal", 4096.0, 1.0), w=("normal", -4096.0, 1.0)))
        parity.compare_grads(d, {k: got[k] for k in PARAMS if k in got}, ref, rtol=RTOL)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_depthwise_masked_taps(dtype):
    for i, d in enumerate(DEPTHWISE):
        d = dict(d, mode="parallel", dtype=dtype)
        t = draw_depthwise(d, 5000 + i)
        for name, v in (("w", np.inf), ("w2", -np.inf)):
            t[name].reshape(-1, 9)[:, [0, 2, 6, 8] if name == "w" else [1, 3, 5, 7]] = v
        got, ref = depthwise(d, t)
        parity.compare_grads(d, {k: got[k] for k in PARAMS}, ref, rtol=RTOL)
