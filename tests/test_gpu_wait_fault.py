"""A step kernel whose bounded wait ran out sets a fault word in the work buffer, and lbm_reduce
answers with an error of its own. No wait is made to run out here: the test writes the word."""
import pytest
import torch

from workloads.params import LBMParams

pytestmark = pytest.mark.gpu

WORD = 0x57414954                     # what the kernels write


@pytest.mark.parametrize("p,steps", [(LBMParams(128, 96, 96), 4),                          # two steps a pass
                                     (LBMParams(512, 243, 242, flow=True, wall_z=True), 1)],  # loads staged by TMA
                         ids=["two-steps", "tma"])
def test_fault_word_becomes_an_error_status(p, steps):
    from paper_2409_03401_gb300 import LBMError, Simulation, _lib
    phi = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
    phi[p.nz // 2] = 1.0
    c = torch.full_like(phi, 0.3)
    sim = Simulation(p, phi, c, c, device="cuda")
    word = sim.work[-256:].view(torch.int32)[2 * _lib.NRED:2 * _lib.NRED + 1]     # behind the sums
    word.fill_(WORD)                  # before a kernel that waits: not the library's
    sim.sums()
    sim.step(steps)                   # clears it
    sim.sums()
    assert int(word) == 0
    word.fill_(WORD)
    for _ in range(2):                # it stays
        with pytest.raises(LBMError, match="wait") as e:
            sim.sums(raise_unstable=False)
        assert e.value.status == _lib.LBM_ERR_CUDA
        sim.step(steps)
    word.zero_()
    sim.sums()
