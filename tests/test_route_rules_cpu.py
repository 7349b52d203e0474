"""Which kernels a step runs on, by size and shape: the answers of the library's rules.

The rules go by what the kernels cost, which depends on the shape of a box, not on its number
of nodes alone: the boxes here were measured on both sides. No device is needed: a context is
bound without touching its buffers.
"""
import ctypes

import pytest

from workloads.params import LBMParams


def _lib():
    from paper_2409_03401_gb300 import _lib as m
    return m, m.load()


@pytest.mark.parametrize("shape,bgk,mrt", [
    ((512, 512, 512), 2, 2), ((384, 384, 384), 2, 2), ((2048, 128, 128), 2, 2), ((4096, 45, 200), 2, 2),
    ((512, 243, 242), 2, 1), ((800, 96, 400), 2, 1), ((256, 256, 458), 1, 1), ((192, 192, 1024), 1, 1),
    ((128, 2048, 128), 1, 1), ((128, 128, 2048), 1, 1), ((64, 700, 671), 1, 1), ((1024, 32, 917), 1, 1),
    ((68, 500, 900), 1, 1), ((4096, 4096, 2), 1, 1), ((510, 512, 512), 1, 1), ((256, 256, 256), 1, 1)])
def test_tma_staged_step_where_its_end_tiles_are_few(shape, bgk, mrt):
    # two launches a step: the pass for phi of the lattice's ends and the TMA-staged kernel
    m, lib = _lib()
    for collision, want in (("BGK", bgk), ("TRT", bgk), ("MRT", mrt)):
        cp = m.make_params(LBMParams(*shape, flow=True, collision=collision))
        ctx = ctypes.c_void_p()
        m.check(lib.lbm_attach(ctypes.byref(cp), ctypes.c_void_p(1 << 20), ctypes.c_void_p(1 << 21), 0, None,
                               ctypes.byref(ctx)))
        assert lib.lbm_kernels_per_step(ctx) == want, (shape, collision)
        lib.lbm_destroy(ctx)
