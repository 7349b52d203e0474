"""Kernels chosen by the shape of a box against the general ones, bit for bit, in boxes that the
rules give them: for the TMA-staged flow step ragged and whole tiles of 32 x 15 nodes, many columns
of tiles and few, thin boxes; for two steps a pass in 3D boxes of whole and ragged tiles of 28 x 14
nodes, narrower than a tile in x, and of few planes; in 2D rows of few windows of 28 nodes, whose warps
go on with the next chunk of rows."""
import ctypes

import pytest
import torch

from workloads.params import LBMParams

pytestmark = pytest.mark.gpu


def _inputs(p, seed=7):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = [torch.rand(p.shape, generator=g, device="cuda", dtype=torch.float64) for _ in range(3)]
    return r[0], 0.3 + 0.1 * r[1], 0.3 + 0.1 * r[2]


@pytest.mark.parametrize("shape", [(2044, 131, 113), (1000, 150, 201), (4096, 45, 163), (2052, 1841, 8)])
@pytest.mark.parametrize("collision,wall_z", [("BGK", True), ("BGK", False), ("TRT", False), ("MRT", True)])
def test_tma_staged_flow_step_matches_the_fused_kernel(shape, collision, wall_z):
    from paper_2409_03401_gb300 import Simulation, _lib
    lib = _lib.load()
    p = LBMParams(*shape, flow=True, collision=collision, wall_z=wall_z)
    f = _inputs(p)
    a, b = (Simulation(p, *f, device="cuda") for _ in range(2))
    assert a.kernels_per_step == 2
    a.step(3)
    cp = _lib.make_params(p)
    copy = lib.lbm_copy_bytes(ctypes.byref(cp))
    at = [ctypes.c_void_p(b.state.data_ptr()), ctypes.c_void_p(b.state.data_ptr() + copy)]
    for t in range(3):
        _lib.check(lib.lbm_step_buffers(ctypes.byref(cp), at[t % 2], at[1 - t % 2], t, None,
                                        ctypes.c_void_p(b.stream.cuda_stream)))
    fa, fb = a.fields(), Simulation.attach(p, b.state, 3).fields()
    for k in fa:
        assert torch.equal(fa[k], fb[k]), k


@pytest.mark.parametrize("shape", [(28, 14, 2600), (16, 512, 128), (15, 288, 260), (513, 512, 8), (85, 43, 4000)])
@pytest.mark.parametrize("wall_x,wall_z", [(False, False), (True, True)])
def test_two_steps_a_pass_match_single_steps(shape, wall_x, wall_z):
    from paper_2409_03401_gb300 import Simulation, _lib
    lib = _lib.load()
    p = LBMParams(*shape, wall_x=wall_x, wall_z=wall_z)
    f = _inputs(p)
    a, b = (Simulation(p, *f, device="cuda") for _ in range(2))
    assert lib.lbm_step_scratch_bytes(ctypes.byref(a._cp)) > 0
    for n in (4, 1, 7):
        a.step(n)
        _lib.check(lib.lbm_step(b._ctx, n), b._ctx)
        fa, fb = a.fields(), b.fields()
        for k in fa:
            assert torch.equal(fa[k], fb[k]), k


@pytest.mark.parametrize("shape", [(1, 700), (27, 1300), (28, 2503), (29, 999), (56, 5000), (57, 3001), (113, 4500), (139, 640),
                                   (240, 1057)])
@pytest.mark.parametrize("kw", [dict(lattice="D2Q9"), dict(lattice="D2Q5"), dict(lattice="D2Q5", wall_x=True)], ids=str)
def test_folded_two_steps_a_pass_match_single_steps(shape, kw):
    from paper_2409_03401_gb300 import Simulation, _lib
    lib = _lib.load()
    p = LBMParams(*shape, 1, **kw)
    f = _inputs(p)
    a, b = (Simulation(p, *f, device="cuda") for _ in range(2))
    assert lib.lbm_step_scratch_bytes(ctypes.byref(a._cp)) > 0
    for n in (4, 1, 7, 8):
        a.step(n)
        _lib.check(lib.lbm_step(b._ctx, n), b._ctx)
        fa, fb = a.fields(), b.fields()
        for k in fa:
            assert torch.equal(fa[k], fb[k]), k
