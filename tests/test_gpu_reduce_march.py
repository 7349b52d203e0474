"""The diagnostics of flow lattices in one read of the state against the fields themselves.

Every sum is compared with the FP64 sum of the same field as lbm_fields writes it. The kernel
adds float pairs (error at most n 2^-47 of the sum of magnitudes for n terms a thread, n below
4096 here: 3e-11) of values that both kernels compute in FP32 with the same formulas; where the
compiler fuses other multiply-adds a value moves by a few units in the last place, so sums are
held to 1e-6 of the sum of magnitudes and max |u| to 1e-5. The droplet count is exact: the
Euler characteristic of the same phi >= 1/2 set. Shapes: tile edges (32 x 8), one-node extents,
several chunks of planes, walls in x and z, both layouts, odd and even time levels.
"""
import pytest
import torch

from oracle.measure import euler_characteristic
from workloads.params import LBMParams

pytestmark = pytest.mark.gpu

# (96, 80, 80) and the shapes after it are read by the marching kernels (FP32 and 16 bits but the
# last, FP32), those before it, small, thin or flat, in separate passes
SHAPES = [(33, 9, 37), (40, 1, 6), (70, 30, 1), (33, 135, 137), (1, 801, 750), (800, 1, 751), (801, 750, 1),
          (96, 80, 80), (125, 101, 61), (126, 94, 67), (1213, 510, 3)]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("wall_x,wall_z", [(False, True), (True, False)])
def test_sums_match_the_fields(storage, inplace, shape, wall_x, wall_z):
    from paper_2409_03401_gb300 import Simulation
    p = LBMParams(*shape, flow=True, storage=storage, inplace=inplace, wall_x=wall_x, wall_z=wall_z)
    g = torch.Generator(device="cuda").manual_seed(11)
    r = [torch.rand(p.shape, generator=g, device="cuda", dtype=torch.float64) for _ in range(3)]
    sim = Simulation(p, r[0], 0.3 + 0.1 * r[1], 0.3 + 0.1 * r[2], device="cuda")
    for _ in range(3):
        f = {k: v.double() for k, v in sim.fields().items()}
        s = sim.sums()
        for k in ("phi", "cA", "cB", "p", "S"):
            assert abs(s[k] - float(f[k].sum())) <= 1e-6 * float(f[k].abs().sum()) + 1e-30, k
        assert abs(s["g"] - float((f["phi"] - 0.5 * f["S"]).sum())) <= 1e-6 * float(f["phi"].abs().sum())
        inter = 4.0 / p.W * f["phi"] * (1 - f["phi"])
        assert abs(s["interface"] - float(inter.sum())) <= 1e-6 * float(inter.abs().sum())
        umax = float(torch.sqrt(f["ux"] ** 2 + f["uy"] ** 2 + f["uz"] ** 2).max())
        assert abs(s["umax"] - umax) <= 1e-5 * umax
        assert s["nonfinite"] == 0
        if p.nz > 1 and p.nodes < 700000:      # the oracle counts nz = 1 as a 2D lattice
            assert s["euler"] == euler_characteristic(f["phi"].cpu().numpy(), walls=(wall_x, False, wall_z))
        sim.step(1)
