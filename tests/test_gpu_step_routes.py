"""The ways a step can run give the same fields, bit for bit.

A two-buffer flow step runs as the fused kernel or as a phi pass with the per-node pull step,
chosen by storage and size; lbm_step_buffers always takes the fused kernel. The sizes lie
around the tiles of the fused kernel (32 x 8 nodes, chunks of up to 32 planes), around the
widths of the per-node blocks, and on both sides of the size where the choice changes. Equality
is exact: both sides do the same arithmetic at every node.
"""
import ctypes

import pytest
import torch

from workloads.params import LBMParams

pytestmark = pytest.mark.gpu


def _inputs(p, seed=7):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = [torch.rand(p.shape, generator=g, device="cuda", dtype=torch.float64) for _ in range(3)]
    return r[0], 0.3 + 0.1 * r[1], 0.3 + 0.1 * r[2]


def _same(a, b):
    for k in a:
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("storage", ["f16", "bf16", "f32", "f64"])
@pytest.mark.parametrize("shape", [(33, 9, 5), (64, 8, 33), (30, 17, 34), (96, 20, 3), (1, 1, 1), (150, 26, 2)])
@pytest.mark.parametrize("collision,wall_z", [("BGK", True), ("TRT", False), ("MRT", True)])
def test_two_buffer_flow_step_matches_the_fused_kernel(storage, shape, collision, wall_z):
    _compare_with_fused(LBMParams(*shape, flow=True, storage=storage, collision=collision, wall_z=wall_z), 5)


def test_fp32_flow_step_on_both_sides_of_the_size_rule():
    _compare_with_fused(LBMParams(100, 75, 79, flow=True, wall_z=True), 4)       # 592,500 nodes: two passes
    _compare_with_fused(LBMParams(100, 75, 81, flow=True, wall_z=True), 4)       # 607,500: the fused kernel


def _compare_with_fused(p, steps):
    from paper_2409_03401_gb300 import Simulation, _lib
    lib = _lib.load()
    f = _inputs(p)
    a, b = (Simulation(p, *f, device="cuda") for _ in range(2))
    a.step(steps)
    cp = _lib.make_params(p)
    copy = lib.lbm_copy_bytes(ctypes.byref(cp))
    at = [ctypes.c_void_p(b.state.data_ptr()), ctypes.c_void_p(b.state.data_ptr() + copy)]
    for t in range(steps):
        _lib.check(lib.lbm_step_buffers(ctypes.byref(cp), at[t % 2], at[1 - t % 2], t, None,
                                        ctypes.c_void_p(b.stream.cuda_stream)))
    _same(a.fields(), Simulation.attach(p, b.state, steps).fields())
