"""The replays of the winner-emitting loops bound the kernels they stand for: compound, whose work is a part of parallel's,
is no slower, and neither kernel outruns its own replay."""
import pytest
import torch

from paper_2504_06881_b200 import inputs, tconv

pytestmark = pytest.mark.gpu


def best_ms(f, n=5):
    f()
    ms = []
    for _ in range(n):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        f()
        e1.record()
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    return min(ms)


def test_winner_replays():
    sink = torch.zeros(4, device="cuda")
    ids, i = {}, 0
    while tconv.tconv_alu_probe_name(i) is not None:
        ids[tconv.tconv_alu_probe_name(i)] = i
        i += 1
    run = lambda name: tconv.tconv_alu_probe(ids[name], 2000, sink)
    rate = {m: max(run(n) / best_ms(lambda: run(n)) for n in (f"f32_win_{m}", f"f32_win_{m}_fb")) for m in ("compound", "parallel")}
    assert rate["compound"] >= 0.98 * rate["parallel"], rate
    for mode in rate:
        d = dict(inputs.layer(32, 64, 32, 32, 64, pad=1), mode=mode, chan="sum", dtype="f32")
        t = {k: torch.from_numpy(v).cuda() for k, v in inputs.draw(d, 3900).items()}
        w2 = t["w2"] if mode == "parallel" else None
        fwd = lambda: tconv.forward(d, t["x"], t["w"], w2, t["alpha"], t["beta"], t["bias"], want_winners=True)
        OH, OW = inputs.output_hw(d)
        got = d["N"] * d["C"] * d["K"] * OH * OW * 9 / best_ms(fwd)
        assert got <= rate[mode], (mode, got, rate)
