"""Winners of the fp32 Sum forms where they can go wrong: a lone winner at every tap of every window, ties of two
taps, constant sums, sums from 2^-120 to 2^100, sums of finite inputs that overflow to an infinity in one tap of a
window and in all of them, padding that never wins."""
import numpy as np
import pytest
import torch

from oracle import tconv_oracle as ora
from paper_2504_06881_b200 import inputs, tconv
import parity
import test_gpu_depthwise

pytestmark = pytest.mark.gpu

L = inputs.layer
WINDOWS = [dict(R=1, S=3, pad=(0, 1)), dict(R=3, S=3, pad=1), dict(R=3, S=3, pad=1, stride=2), dict(R=3, S=3, pad=2, dil=2),
           dict(R=5, S=5, pad=2)]
MODES = [("compound", "sum"), ("parallel", "sum"), ("max_plus", "sum"), ("min_plus", "sum")]


def check(d, t):
    _, _, winners = parity.check_forward(d, t)
    assert tconv.tconv_last_kernel().startswith("fwd_tiled_f32")


@pytest.mark.parametrize("mode,chan", MODES)
@pytest.mark.parametrize("window", WINDOWS, ids=lambda w: f"{w['R']}x{w['S']}s{w.get('stride', 1)}d{w.get('dil', 1)}")
def test_winning_taps(mode, chan, window):
    RS = window["R"] * window["S"]
    d = dict(L(2, 9, 9 if window["R"] > 1 else 1, 20, 2 * RS + 1, **window), mode=mode, chan=chan, dtype="f32")
    t = inputs.draw(d, 2500)
    rng = np.random.RandomState(2501)
    # output channel k < RS: tap k wins by its weight alone (max, then min in the other half); two taps tie in k >= RS
    for k in range(d["K"]):
        for name, sign in (("w", -1.0), ("w2", 1.0)) if mode == "parallel" else (("w", 1.0 if mode != "min_plus" else -1.0),):
            flat = t[name][k].reshape(d["C"], RS)
            flat[:] = 0.0
            flat[:, k % RS] = sign * 64.0
            if k >= RS:
                flat[:, rng.randint(RS)] = sign * 64.0
    t["x"] = rng.randint(-2, 3, t["x"].shape).astype(np.float32)
    check(d, t)
    # few distinct sums: ties everywhere; then the same sums at 2^100 (their differences as large) and 2^-120
    for scale in (1.0, 2.0 ** 100, 2.0 ** -120):
        for name in ("x", "w", "w2"):
            t[name] = (rng.randint(-1, 2, t[name].shape) * scale).astype(np.float32)
        check(d, t)
    if window.get("dil", 1) == 1 and window["R"] > 1:
        check(dict(d, pad_mode="neutral"), t)


@pytest.mark.parametrize("mode,chan", MODES)
@pytest.mark.parametrize("window", WINDOWS, ids=lambda w: f"{w['R']}x{w['S']}s{w.get('stride', 1)}d{w.get('dil', 1)}")
def test_sums_that_overflow(mode, chan, window):
    """All infinities of a layer have one sign and alpha = beta = 1, so that no output is a NaN."""
    RS = window["R"] * window["S"]
    d = dict(L(1, 3, 9 if window["R"] > 1 else 1, 20, RS + 1, **window), mode=mode, chan=chan, dtype="f32")
    t = inputs.draw(d, 2502)
    for name in ("alpha", "beta"):
        t[name][:] = 1.0
    for sign in (1.0, -1.0):
        t["x"][:] = sign * 2.0e38
        for name in ("w", "w2"):
            t[name][:] = 0.0
            for k in range(RS):                              # tap k alone, then (channel RS) every tap
                t[name][k].reshape(d["C"], RS)[:, k] = sign * 2.0e38
            if RS <= 16:        # (wide codes are compared with Max / Min layers, whose winner of such a window is none)
                t[name][RS] = sign * 2.0e38
        _, y, _ = parity.check_forward(d, t)
        assert np.isinf(y.cpu().numpy()).any()
        assert tconv.tconv_last_kernel().startswith("fwd_tiled_f32")


@pytest.mark.parametrize("mode", ["compound", "parallel", "max_plus", "min_plus"])
@pytest.mark.parametrize("stride", [1, 2])
def test_depthwise_sums_that_overflow(mode, stride):
    """Channel k of nine: tap k overflows; the last channel: every tap."""
    d = inputs.layer(2, 10, 9, 17, 10, 3, 3, mode=mode, stride=stride, pad=1)
    par, two = mode == "parallel", mode in ("compound", "parallel")
    t = test_gpu_depthwise.draw(d, 2503)
    dev = lambda name, used=True: torch.from_numpy(t[name]).cuda() if used else None
    t["alpha"][:], t["beta"][:] = 1.0, 1.0
    for sign in (1.0, -1.0):
        t["x"][:] = sign * 2.0e38
        for name in ("w", "w2"):
            t[name][:] = 0.0
            for k in range(9):
                t[name][k].reshape(9)[k] = sign * 2.0e38
            t[name][9] = sign * 2.0e38
        ref = ora.depthwise_forward(d, t["x"], t["w"], t["w2"] if par else None, t["alpha"] if two else None,
                                    t["beta"] if two else None, t["bias"])
        y, win = tconv.dw_forward(d, dev("x"), dev("w"), dev("w2", par), dev("alpha", two), dev("beta", two), dev("bias"),
                                  want_winners=True)
        assert np.isinf(ref["y"]).any() and parity.same_bits(y.cpu().numpy(), ref["y"]).all()
        assert np.array_equal(win.cpu().numpy(), ref["codes"])
