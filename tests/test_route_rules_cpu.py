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


# boxes and the measured time of a single step over that of two steps a pass
@pytest.mark.parametrize("shape,ratio", [
    ((256, 256, 256), 1.43), ((128, 128, 128), 1.29), ((128, 96, 96), 1.15), ((150, 84, 80), 1.01), ((28, 14, 4000), 2.04),
    ((16, 512, 128), 2.36), ((15, 288, 3900), 2.56), ((64, 64, 4096), 1.24), ((512, 512, 8), 1.27), ((85, 43, 4000), 1.16),
    ((1024, 1024, 1), 0.65), ((1024, 1, 1024), 0.15), ((29, 15, 2400), 0.68), ((29, 15, 38000), 0.85), ((57, 29, 1000), 0.85),
    ((512, 16, 128), 0.76), ((64, 64, 256), 0.88), ((60, 60, 300), 0.81), ((101, 101, 101), 0.95), ((207, 691, 8), 0.89),
    ((96, 96, 96), 0.88)])
def test_two_steps_a_pass_where_the_box_suits_the_tiles(shape, ratio):
    m, lib = _lib()
    cp = ctypes.byref(m.make_params(LBMParams(*shape)))
    want = lib.lbm_copy_bytes(cp) if ratio > 1 else 0
    assert lib.lbm_step_scratch_bytes(cp) == want, shape


@pytest.mark.parametrize("lattice,shape,ratio", [
    ("D2Q9", (4096, 4096), 1.71), ("D2Q9", (512, 512), 0.99), ("D2Q9", (29, 20000), 1.04), ("D2Q9", (120, 2563), 1.03),
    ("D2Q9", (28, 20000), 1.59), ("D2Q9", (64, 16384), 1.37), ("D2Q9", (768, 768), 1.09), ("D2Q9", (128, 3125), 1.05),
    ("D2Q9", (64, 4096), 0.87), ("D2Q9", (64, 8192), 0.88), ("D2Q9", (256, 2343), 0.91), ("D2Q9", (384, 1562), 0.96),
    ("D2Q9", (48, 48), 1.28), ("D2Q5", (2048, 512), 1.03), ("D2Q5", (1024, 1024), 0.96), ("D2Q5", (256, 4687), 0.88),
    ("D2Q5", (96, 12500), 0.92), ("D2Q5", (64, 16384), 1.22), ("D2Q5", (124, 2842), 1.21), ("D2Q5", (4096, 4096), 1.58)])
def test_two_steps_a_pass_in_2d(lattice, shape, ratio):
    m, lib = _lib()
    cp = ctypes.byref(m.make_params(LBMParams(*shape, 1, lattice=lattice)))
    want = lib.lbm_copy_bytes(cp) if ratio > 1 else 0
    assert lib.lbm_step_scratch_bytes(cp) == want, shape
