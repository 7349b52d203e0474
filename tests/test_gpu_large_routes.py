"""The kernels that only larger lattices reach, against something that does not share their code.

* FP32 flow steps of 600,000 nodes and more run as the fused kernel, and their fields and sums come
  from a march through the lattice: both against the FP64 oracle, in ragged boxes (tiles of 32 x 8,
  chunks of planes), two copies and in place, odd and even time levels, walls in x and z.
* The droplet count of the march in ragged boxes, with every combination of walls, against the
  Euler characteristic of phi >= 1/2 on the host.
* Warps inside the lattice take other addresses than those at its ends: a periodic lattice moved by
  some nodes gives the same fields, moved, bit for bit (every node's neighbours are the same).
* Out-of-bounds writes: guard regions around state, work and scratch of these kernels.
"""
import ctypes

import pytest
import torch

from oracle.lbm import OracleLBM
from oracle.measure import euler_characteristic
from parity import TOL, rel_linf
from workloads import configs
from workloads.params import LBMParams

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(61, 101, 125), (67, 94, 126)])          # nz, ny, nx
@pytest.mark.parametrize("kw", [dict(), dict(wall_x=True), dict(wall_z=False, collision="TRT"), dict(collision="MRT"),
                                dict(inplace=True), dict(inplace=True, wall_x=True, wall_z=False)], ids=str)
def test_fused_steps_and_marched_fields_match_the_oracle(shape, kw):
    from paper_2409_03401_gb300 import Simulation
    p, fields = configs.sedimentation(shape=shape, fraction=0.06, r=(4.0, 9.0))
    p = p.with_(nu=0.05, **kw)
    f = fields()
    sim, o = Simulation(p, *f, device="cuda"), OracleLBM(p)
    o.init(*f)
    for n in (1, 2, 1):                                                      # time levels 1, 3, 4
        sim.step(n)
        o.step(n)
        g, r, s = sim.fields(), o.fields(), sim.sums()
        for k in ("phi", "muA", "muB", "cA", "cB", "p", "ux", "uy", "uz"):
            assert rel_linf(g[k], r[k], k) <= TOL["f32"], k
        for k in ("phi", "cA", "cB"):
            assert abs(s[k] - float(r[k].sum())) <= TOL["f32"] * float(r[k].abs().sum()), k
        umax = float(torch.sqrt(r["ux"] ** 2 + r["uy"] ** 2 + r["uz"] ** 2).max())
        assert abs(s["umax"] - umax) <= 3 * TOL["f32"] * umax                # three components
        assert s["nonfinite"] == 0


def _random(p, seed=11):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = [torch.rand(p.shape, generator=g, device="cuda", dtype=torch.float64) for _ in range(3)]
    return r[0], 0.3 + 0.1 * r[1], 0.3 + 0.1 * r[2]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("shape", [(125, 101, 61), (126, 94, 67)])
@pytest.mark.parametrize("wall_x,wall_z", [(False, True), (True, False), (True, True), (False, False)])
def test_marched_droplet_count_in_ragged_boxes(storage, inplace, shape, wall_x, wall_z):
    from paper_2409_03401_gb300 import Simulation
    p = LBMParams(*shape, flow=True, storage=storage, inplace=inplace, wall_x=wall_x, wall_z=wall_z)
    sim = Simulation(p, *_random(p), device="cuda")
    for _ in range(2):
        phi = sim.fields(("phi",))["phi"].double().cpu().numpy()
        assert sim.sums()["euler"] == euler_characteristic(phi, walls=(wall_x, False, wall_z))
        sim.step(1)


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("kw", [dict(inplace=True), dict(inplace=True, collision="MRT"), dict(lattice="D3Q19"),
                                dict(lattice="D3Q19", inplace=True), dict(lattice="D3Q19", flow=False)], ids=str)
def test_fields_move_with_the_lattice(storage, kw):
    from paper_2409_03401_gb300 import Simulation
    p = LBMParams(130, 9, 7, flow=kw.get("flow", True), storage=storage, **{k: v for k, v in kw.items() if k != "flow"})
    f = _random(p)
    move = dict(shifts=(3, 4, 41), dims=(0, 1, 2))
    a = Simulation(p, *f, device="cuda")
    b = Simulation(p, *[torch.roll(t, **move) for t in f], device="cuda")
    for n in (1, 1, 2):
        a.step(n)
        b.step(n)
        fa, fb = a.fields(), b.fields()
        for k in fa:
            assert torch.equal(torch.roll(fa[k], **move), fb[k]), k


GUARD, FILL = 1 << 16, 0xA5


@pytest.mark.parametrize("p", [
    LBMParams(125, 101, 61, flow=True, wall_z=True), LBMParams(125, 101, 61, flow=True, inplace=True, wall_x=True),
    LBMParams(125, 101, 61, flow=True, storage="f16", wall_z=True), LBMParams(125, 101, 61, flow=True, storage="bf16"),
    LBMParams(125, 101, 61, flow=True, collision="MRT"), LBMParams(1000, 150, 201, flow=True, wall_z=True),
    LBMParams(1004, 151, 201, flow=True, collision="MRT"), LBMParams(150, 85, 80), LBMParams(15, 288, 260, wall_z=True),
    LBMParams(301, 300, 1, lattice="D2Q9"), LBMParams(113, 4500, 1, lattice="D2Q5", wall_x=True)],
    ids=lambda p: f"{p.nx}x{p.ny}x{p.nz}-{p.lattice}-{p.storage}-{'flow' if p.flow else 'no flow'}-{p.collision}")
def test_no_write_outside_the_given_buffers(p):
    from paper_2409_03401_gb300 import _lib
    lib = _lib.load()
    cp = _lib.make_params(p)
    sizes = [lib.lbm_state_bytes(ctypes.byref(cp)), lib.lbm_work_bytes(ctypes.byref(cp)),
             lib.lbm_step_scratch_bytes(ctypes.byref(cp))]
    at, end = [], GUARD
    for n in sizes:
        at.append(end)
        end += (n + 255) // 256 * 256 + GUARD
    buf = torch.full((end,), FILL, dtype=torch.uint8, device="cuda")
    state, work, scratch = (ctypes.c_void_p(buf.data_ptr() + o) for o in at)
    rdt = torch.float64 if p.storage == "f64" else torch.float32
    outs = [torch.full((p.nodes + 2 * GUARD,), 12345.0, dtype=rdt, device="cuda") for _ in range(_lib.NFIELDS)]
    ptrs = (ctypes.c_void_p * _lib.NFIELDS)(*[t.data_ptr() + GUARD * t.element_size() for t in outs])
    f = [t.contiguous() for t in _random(p)]
    ctx = ctypes.c_void_p()
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    _lib.check(lib.lbm_init(ctypes.byref(cp), state, work, *[ctypes.c_void_p(t.data_ptr()) for t in f], stream,
                            ctypes.byref(ctx)))
    try:
        red = (ctypes.c_double * _lib.NRED)()
        for n in (1, 6, 4):                           # odd and even time levels
            _lib.check(lib.lbm_step_scratch(ctx, n, scratch, sizes[2]), ctx)
            _lib.check(lib.lbm_fields(ctx, ptrs), ctx)
            _lib.check(lib.lbm_reduce(ctx, red), ctx)
    finally:
        lib.lbm_destroy(ctx)
    torch.cuda.synchronize()
    for a, b in zip([0] + [o + n for o, n in zip(at, sizes)], at + [end]):
        assert bool((buf[a:b] == FILL).all()), (a, b)
    for name, t in zip(_lib.FIELDS, outs):
        assert bool((t[:GUARD] == 12345.0).all()) and bool((t[GUARD + p.nodes:] == 12345.0).all()), name
        assert not bool((t[GUARD:GUARD + p.nodes] == 12345.0).any()), name
