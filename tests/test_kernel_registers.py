"""Kernel instances whose speed hangs on how many blocks an SM holds stay within the registers that allows, without
spilling to get there."""
from nvcc_probe import resources

FILE = 65536     # registers of an SM


def test_finishing_sum():
    """Eight blocks of 256 threads."""
    got = resources("tconv_bwd_sum.cuh", ["bwd_sum_finish_kernel<1>", "bwd_sum_finish_kernel<16>"])
    assert all(regs <= FILE // 256 // 8 and spilled <= 64 for regs, spilled in got.values()), got
