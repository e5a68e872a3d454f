"""The Sum-form backward takes its tile kernels for maps of any size that their 31-bit counts allow.  (They keep the
inputs' regions of all tiles in the workspace, the any-shape kernels only sums of grad_y.)"""
import pytest
import torch

from paper_2504_06881_b200 import inputs, tconv

L = inputs.layer


@pytest.mark.parametrize("d", [
    L(1, 2, 4096, 4096, 4, pad=1, mode="compound"),              # 1.7e7 positions
    L(1, 2, 2048, 2048, 256, pad=1, mode="parallel"),            # 1.1e9 outputs of one image
    L(1, 128, 1024, 1024, 128, pad=1, mode="compound"),          # 1.7e10 winners of one image
    L(1, 1, 45000, 45000, 1, pad=1, mode="max_plus", chan="sum"),
])
def test_large_maps_keep_the_tile_kernels(d):
    free = tconv.tconv_workspace_bytes(d, True) - tconv.tconv_winner_bytes(d)
    assert free >= 4 * d["N"] * d["C"] * d["H"] * d["W"]


@pytest.mark.gpu
@pytest.mark.parametrize("K,dtype,rtol", [(260, "f32", 1e-5), (1028, "bf16", 8e-3)])      # (bf16 grad_x: one rounding step)
def test_outputs_of_one_image_beyond_a_billion(K, dtype, rtol):
    """The last four of K output channels at 2048 x 2048 against a layer of these four alone; 1028 channels are more
    gradients than a 32-bit count."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    dt = tconv.TORCH_DTYPE[dtype]
    rand = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    big = L(1, 1, 2048, 2048, K, pad=1, mode="compound", dtype=dtype)
    few = dict(big, K=4)
    x, w, g4 = rand(1, 1, 2048, 2048).to(dt), (rand(K, 1, 3, 3) * 0.3).to(dt), rand(1, 4, 2048, 2048).to(dt)
    al, be = rand(K, 1), rand(K, 1)
    last = lambda t: t[K - 4:].contiguous()
    y4, win4 = tconv.forward(few, x, last(w), None, last(al), last(be), None, want_winners=True)
    ref = tconv.backward(few, x, last(w), g4, None, last(al), last(be), win4)
    y, win = tconv.forward(big, x, w, None, al, be, None, want_winners=True)
    assert torch.equal(y[:, K - 4:], y4) and torch.equal(win[-win4.numel():], win4)
    del y
    g = torch.zeros(1, K, 2048, 2048, device="cuda", dtype=dt)
    g[:, K - 4:] = g4
    got = tconv.backward(big, x, w, g, None, al, be, win)
    assert tconv.tconv_last_kernel() == "bwd_sum"
    assert torch.allclose(got["grad_x"].float(), ref["grad_x"].float(), rtol=rtol, atol=1e-5)
    bound = 1e-5 * float(g4.float().abs().sum()) / 4      # the sums' order: 1e-5 of the sum of |contributions|, |x + w| about 1
    for name in ("grad_w", "grad_alpha", "grad_beta", "grad_bias"):
        assert (got[name][:K - 4] == 0).all(), name
        assert (got[name][K - 4:] - ref[name]).abs().max() <= bound, name
