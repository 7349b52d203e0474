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


@pytest.mark.parametrize("storage", ["f16", "f32", "f64"])
@pytest.mark.parametrize("shape", [(20, 128, 64), (20, 130, 70)])      # 8192 and 9100 narrow blocks
def test_phi_pass_of_many_narrow_blocks(storage, shape):
    _compare_with_fused(LBMParams(*shape, flow=True, storage=storage), 5)


@pytest.mark.parametrize("shape", [(64, 700, 671), (100, 601, 500), (1024, 32, 917), (512, 243, 242)])
@pytest.mark.parametrize("collision,wall_z", [("BGK", True), ("BGK", False), ("TRT", False), ("MRT", True)])
def test_tma_staged_flow_step_matches_the_fused_kernel(shape, collision, wall_z):
    # from 30 million nodes on, rows of whole 16-byte pieces: the step's loads come by tensor copies,
    # the lattice's ends apart; tiles of 32 x 15 nodes, the last ones overlapping, several chunks
    _compare_with_fused(LBMParams(*shape, flow=True, collision=collision, wall_z=wall_z), 3)


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


def _two_against_single(p, steps=(8, 1, 9, 7, 4)):
    # two steps per pass (the scratch buffer lent here whatever the lattice's size) and single steps
    from paper_2409_03401_gb300 import Simulation, _lib
    lib = _lib.load()
    f = _inputs(p)
    a, b = (Simulation(p, *f, device="cuda") for _ in range(2))
    scratch = torch.empty(lib.lbm_copy_bytes(ctypes.byref(a._cp)), dtype=torch.uint8, device="cuda")
    for n in steps:
        _lib.check(lib.lbm_step_scratch(a._ctx, n, ctypes.c_void_p(scratch.data_ptr()), scratch.numel()), a._ctx)
        _lib.check(lib.lbm_step(b._ctx, n), b._ctx)
        assert a.t == b.t
        _same(a.fields(), b.fields())


@pytest.mark.parametrize("wall_x,wall_z", [(False, False), (True, False), (False, True), (True, True)])
def test_two_steps_per_pass_match_single_steps_3d(wall_x, wall_z):
    # 1,008,000 nodes, just over the size rule: several 28 x 14 tiles with ragged ends
    _two_against_single(LBMParams(150, 84, 80, wall_x=wall_x, wall_z=wall_z), (8, 1, 7))


@pytest.mark.parametrize("nx", [1, 2, 27, 28, 29, 57, 512])
@pytest.mark.parametrize("ny", [1, 3, 90])
def test_two_steps_per_pass_match_single_steps_2d(nx, ny):
    # window edges (28 nodes), lattices narrower than a window, one-row lattices, walls in x
    _two_against_single(LBMParams(nx, ny, 1, lattice="D2Q9"))
    _two_against_single(LBMParams(nx, ny, 1, lattice="D2Q5"))
    _two_against_single(LBMParams(nx, ny, 1, lattice="D2Q5", wall_x=True))


def test_step_scratch_takes_what_it_can_use_and_no_more():
    from paper_2409_03401_gb300 import LBMError, Simulation, _lib
    lib = _lib.load()
    p = LBMParams(128, 96, 96)
    f = _inputs(p)
    a, b = (Simulation(p, *f, device="cuda") for _ in range(2))
    need = lib.lbm_step_scratch_bytes(ctypes.byref(a._cp))
    assert need == lib.lbm_copy_bytes(ctypes.byref(a._cp)) > 0
    for q in (p.with_(flow=True), p.with_(storage="f64"), p.with_(storage="f16"), p.with_(lattice="D3Q19"),
              p.with_(nx=32), LBMParams(64, 64, 1, lattice="D2Q9", wall_x=True)):
        assert lib.lbm_step_scratch_bytes(ctypes.byref(_lib.make_params(q))) == 0
    guard = 1 << 16
    buf = torch.full((need + 2 * guard,), 0xA5, dtype=torch.uint8, device="cuda")
    with pytest.raises(LBMError):
        _lib.check(lib.lbm_step_scratch(a._ctx, 4, ctypes.c_void_p(buf.data_ptr() + 8), need), a._ctx)
    assert a.t == 0
    short = ctypes.c_void_p(buf.data_ptr() + guard)
    _lib.check(lib.lbm_step_scratch(a._ctx, 5, short, need - 1), a._ctx)         # too small: single steps
    assert bool((buf == 0xA5).all())
    _lib.check(lib.lbm_step_scratch(a._ctx, 6, short, need), a._ctx)
    b.step(3).step(8)
    _same(a.fields(), b.fields())
    assert bool((buf[:guard] == 0xA5).all()) and bool((buf[guard + need:] == 0xA5).all())
    # a stream under capture takes the single steps, and the graph replays them
    s = torch.cuda.Stream()
    c = Simulation(p, *f, device="cuda", stream=s)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        c.step(6)
    g.replay()
    torch.cuda.synchronize()
    d = Simulation(p, *f, device="cuda").step(6)
    _same(c.fields(), d.fields())
