"""Winners of the fp32 Sum forms where they can go wrong: a lone winner at every tap of every window, ties of two
taps, constant sums, sums of any magnitude up to the largest floats, padding that never wins."""
import numpy as np
import pytest

from paper_2504_06881_b200 import inputs, tconv
import parity

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
