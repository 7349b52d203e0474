"""The state copy that Simulation.step borrows for two steps a pass: never where it could harm."""
import pytest
import torch

from workloads.params import LBMParams

pytestmark = pytest.mark.gpu

P = LBMParams(128, 96, 96)


def _sim(**kw):
    from paper_2409_03401_gb300 import Simulation
    g = torch.Generator(device="cuda").manual_seed(3)
    r = [torch.rand(P.shape, generator=g, device="cuda", dtype=torch.float64) for _ in range(3)]
    return Simulation(P, r[0], 0.3 + 0.1 * r[1], 0.3 + 0.1 * r[2], device="cuda", **kw)


def _same(a, b):
    fa, fb = a.fields(), b.fields()
    for k in fa:
        assert torch.equal(fa[k], fb[k]), k


def test_step_while_another_stream_is_captured():
    a, b = _sim(stream=torch.cuda.Stream()), _sim()
    warm = _sim()
    warm.step(8), warm.step(1), warm.close()
    del warm
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):                # empties torch's cache first, captures in the global mode
        x += 1
        a.step(9)                            # queued on its own stream, not captured
        x += 1
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 2.0
    b.step(9)
    assert a.t == b.t == 9
    _same(a, b)


def test_no_memory_is_asked_for_once(monkeypatch):
    a, b = _sim(), _sim()
    empty, asked = torch.empty, []

    def refuse(*size, **kw):
        if kw.get("dtype") == torch.uint8:
            asked.append(size)
            raise torch.cuda.OutOfMemoryError("none left")
        return empty(*size, **kw)

    monkeypatch.setattr(torch, "empty", refuse)
    a.step(8).step(5).step(4)
    monkeypatch.undo()
    assert len(asked) == 1
    b.step(17)
    _same(a, b)


def test_scratch_can_be_declined():
    a, b = _sim(), _sim()
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    a.step(8, scratch=False)
    assert torch.cuda.max_memory_allocated() == before
    b.step(8)
    assert torch.cuda.max_memory_allocated() > before
    _same(a, b)
