"""The TMA-staged flow step against the fused kernel, bit for bit, in boxes that its rule gives it:
ragged and whole tiles of 32 x 15 nodes in x and y, many columns of tiles and few, thin boxes."""
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
