"""Which lattices LD_KERNEL_AUTO steps with the one-launch kernel, without a
GPU: the choice on lattices whose faster kernel was measured to be faster by 5 %
or more, narrow ones, tiles that reach past the lattice, both stencils."""

import ctypes

import pytest

from paper_1609_01479_gb300 import ld

SMALL, REGS, GENERIC = 4, 3, 1


def choice(nx, ny, nz, stencil=7, precision=None, kernel=0):
    fn = getattr(ld.lib(), "_ZN2ld18choose_step_kernelEiiiiii")  # ld::choose_step_kernel
    fn.argtypes, fn.restype = [ctypes.c_int] * 6, ctypes.c_int
    return fn(nx, ny, nz, ld.LD_FP32 if precision is None else precision, ld.STENCILS[stencil], kernel)


# us a step of the one-launch kernel and of the other one
@pytest.mark.parametrize("dims,stencil,small,other", [
    ((4, 4, 16384), 7, 117, 20.8), ((4, 4, 16384), 19, 135, 25.0), ((4, 128, 128), 7, 31.8, 10.3),
    ((4, 91, 90), 7, 16.8, 9.0), ((4, 91, 90), 19, 19.3, 14.4), ((4, 64, 64), 7, 9.7, 8.3),
    ((4, 64, 64), 19, 11.5, 12.4), ((5, 81, 80), 7, 14.3, 9.7), ((8, 45, 45), 7, 5.2, 8.3),
    ((17, 17, 17), 7, 4.9, 8.3), ((20, 57, 57), 7, 8.6, 10.3), ((31, 65, 65), 7, 12.2, 13.9),
    ((33, 33, 33), 7, 8.2, 10.3), ((33, 45, 44), 7, 12.0, 10.3), ((33, 63, 63), 7, 20.0, 14.2),
    ((33, 65, 65), 19, 25.9, 18.5), ((45, 45, 45), 19, 15.0, 16.5), ((50, 61, 47), 7, 17.1, 14.4),
    ((50, 61, 47), 19, 20.4, 18.5), ((100, 51, 51), 7, 28.8, 21.6), ((1000, 5, 7), 7, 6.5, 9.2),
    ((32, 32, 32), 7, 5.9, 14.5), ((96, 96, 24), 7, 19.5, 22.7), ((96, 96, 24), 19, 23.2, 24.7),
    ((32, 128, 64), 7, 22.3, 20.7), ((64, 64, 64), 19, 26.6, 24.7), ((32, 8, 1024), 19, 25.8, 22.2),
])
def test_auto_takes_the_faster_kernel(dims, stencil, small, other):
    nx, ny, nz = dims
    tiled = nx % 32 == 0 and ny % 8 == 0 and nz % 4 == 0
    assert choice(*dims, stencil) == (SMALL if small < other else REGS if tiled else GENERIC)


def test_only_auto_and_only_fp32():
    for precision in (ld.LD_FP64, ld.LD_FP16DEV, ld.LD_BF16DEV):
        assert choice(32, 32, 32, precision=precision) != SMALL
    assert choice(32, 32, 32, kernel=1) == GENERIC and choice(32, 32, 32, kernel=2) == REGS
    assert choice(2048, 1024, 1023) == GENERIC  # 2^31 sites less a plane: the tile count does not overflow
