"""Kernels queued behind one another give what they give one at a time.

Step and adjoint kernels may be set up while the one before still runs. Small lattices are where
several overlap: many steps in one call against the same steps with the stream synchronised
after each, and one call for a segment of the reverse sweep against its kernels one by one. Both
sides run the same kernels, so they are equal bit for bit.
"""
import ctypes

import pytest
import torch

from workloads.params import LBMParams

pytestmark = pytest.mark.gpu


def _inputs(p):
    # one droplet off the middle, with a little noise
    g = torch.Generator(device="cuda").manual_seed(5)
    r = [torch.rand(p.shape, generator=g, device="cuda", dtype=torch.float64) for _ in range(3)]
    d2 = sum((torch.arange(m, device="cuda", dtype=torch.float64) - 0.4 * m).reshape([-1 if i == a else 1 for i in range(3)]) ** 2
             for a, m in enumerate(p.shape) if m > 1)
    phi = 0.5 + 0.5 * torch.tanh((0.25 * max(p.shape) - torch.sqrt(d2)) * 2.0 / 3.0)
    return phi * 0.98 + 0.02 * r[0], 0.3 + 0.01 * r[1], 0.3 + 0.01 * r[2]


@pytest.mark.parametrize("kw", [dict(), dict(inplace=True), dict(storage="f16"), dict(storage="f64"),
                                dict(lattice="D3Q19"), dict(collision="MRT")], ids=str)
@pytest.mark.parametrize("n", [16, 23, 40, 64])
def test_flow_steps_back_to_back_and_one_at_a_time(n, kw):
    from paper_2409_03401_gb300 import Simulation
    p = LBMParams(n, n, n, flow=True, wall_z=True, **kw)
    f = _inputs(p)
    a, b = (Simulation(p, *f, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    a.step(200)
    for _ in range(200):
        b.step(1)
        torch.cuda.synchronize()
    fa, fb = a.fields(), b.fields()
    for k in fa:
        assert bool(torch.isfinite(fa[k]).all()) and torch.equal(fa[k], fb[k]), k


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("shape,lattice", [((16, 16, 16), "D3Q7"), ((33, 18, 21), "D3Q19"), ((90, 40, 1), "D2Q9")])
def test_adjoint_segment_and_its_kernels_one_at_a_time(shape, lattice, storage):
    from paper_2409_03401_gb300 import Simulation, _lib
    lib = _lib.load()
    p = LBMParams(*shape, lattice=lattice, storage=storage)
    cp = ctypes.byref(_lib.make_params(p))
    n = 24
    sim = Simulation(p, *_inputs(p), device="cuda")
    stream = ctypes.c_void_p(sim.stream.cuda_stream)
    copy, lam_bytes = lib.lbm_copy_bytes(cp), lib.lbm_adjoint_bytes(cp)
    g = torch.Generator(device="cuda").manual_seed(2)
    seed = [torch.rand(p.shape, generator=g, device="cuda", dtype=sim.real_dtype) for _ in range(3)]

    def ptr(t, off=0):
        return ctypes.c_void_p(t.data_ptr() + off)

    def bytes_of(k):
        return torch.zeros(k, dtype=torch.uint8, device="cuda")

    start = sim.state.clone()
    sim.step(n)
    out = []
    for single in (False, True):
        ring, lam, tmp = bytes_of(n * copy), bytes_of(lam_bytes), bytes_of(lam_bytes)
        work = bytes_of(lib.lbm_adjoint_work_bytes(cp))
        ring[:copy].copy_(start)
        _lib.check(lib.lbm_adjoint_reset(cp, ptr(work), stream))
        _lib.check(lib.lbm_adjoint_seed(cp, ptr(sim.state), n, *[ptr(t) for t in seed], ptr(lam), ptr(work), stream))
        if not single:
            which = ctypes.c_int(0)
            _lib.check(lib.lbm_adjoint_segment(cp, ptr(ring), 0, n, ptr(lam), ptr(tmp), ptr(work), ptr(sim.work), stream,
                                               ctypes.byref(which)))
            if which.value:
                lam, tmp = tmp, lam
        else:
            for t in range(n - 1):
                _lib.check(lib.lbm_step_buffers(cp, ptr(ring, t * copy), ptr(ring, (t + 1) * copy), t, ptr(sim.work), stream))
                torch.cuda.synchronize()
            for t in reversed(range(n)):
                _lib.check(lib.lbm_adjoint_step(cp, ptr(ring, t * copy), t, ptr(lam), ptr(tmp), ptr(work), stream))
                torch.cuda.synchronize()
                lam, tmp = tmp, lam
        theta = (ctypes.c_double * 5)()
        _lib.check(lib.lbm_adjoint_theta(cp, ptr(work), theta, stream))
        out.append((lam.clone(), list(theta)))
    assert torch.equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
