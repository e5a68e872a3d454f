"""Kernel instances whose speed hangs on how many blocks an SM holds stay within the registers that allows, without
spilling to get there."""
import pytest

from nvcc_probe import resources

FILE = 65536     # registers of an SM


@pytest.mark.parametrize("dtype", ["float", "__nv_bfloat16"])
def test_1d_forward_with_winners(dtype):
    """Four blocks of 128 threads; three at stride 4 with two branches."""
    most = {f"fwd1d_kernel<{dtype}, {st}, {br}, true, false>": FILE // 128 // (3 if st == 4 and br == 3 else 4)
            for st in (1, 2, 4) for br in (1, 3)}
    got = resources("tconv_1d.cuh", list(most))
    assert all(got[k][0] <= most[k] // 8 * 8 for k in most), got


@pytest.mark.parametrize("dtype", ["float", "__nv_bfloat16"])
def test_1d_forward_without_winners(dtype):
    """Four blocks of 128 threads; five with two branches and more blocks than four per SM hold."""
    most = {f"fwd1d_kernel<{dtype}, {st}, {br}, false, {few}>": FILE // 128 // (5 if br >= 2 and few == "false" else 4)
            for st in (1, 2, 4) for br in (1, 2, 3) for few in ("false", "true") if not (dtype == "float" and st == 4)}
    got = resources("tconv_1d.cuh", list(most))
    assert all(got[k][0] <= most[k] // 8 * 8 and got[k][1] <= 32 for k in most), got


@pytest.mark.parametrize("dtype", ["float", "__nv_bfloat16"])
def test_depthwise_parameter_gradients(dtype):
    """Three blocks of 256 threads where they do not spill, two elsewhere: at most 32 bytes."""
    names = [f"dw_bwd_params3_kernel<{dtype}, {br}, {par}, {sw}, {vec}>" for br, par in ((0, "false"), (0, "true"), (2, "false"))
             for sw in (1, 2) for vec in ("true", "false")]
    got = resources("tconv_depthwise.cuh", names)
    assert all(regs <= FILE // 256 // 2 and spilled <= 32 for regs, spilled in got.values()), got
    assert all(got[k][0] <= 80 for k in names if "true, 2" not in k), got


def test_finishing_sum():
    """Eight blocks of 256 threads."""
    got = resources("tconv_bwd_sum.cuh", ["bwd_sum_finish_kernel<1>", "bwd_sum_finish_kernel<16>"])
    assert all(regs <= FILE // 256 // 8 and spilled <= 64 for regs, spilled in got.values()), got
