"""Kernels that may start before the one ahead of them in the stream has ended (they begin with
begin_after_previous, programmatic dependent launch) take no __restrict__ pointers: a const one
lets the compiler use read-only loads, whose data must not change during the kernel's life, and
what such a kernel reads is still being written when its blocks are set up. Read from the source.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_03401_gb300", "csrc")


def _kernels():
    """(name, parameter list, start of the body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\(.*?\)\)?\s*\n)?(\w+)\(([^{]*?)\)\s*\{", src, re.S):
            yield m.group(1), m.group(2), src[m.end():m.end() + 2500].split("__global__")[0]


def test_dependent_kernels_take_no_restrict_pointers():
    early = {name: params for name, params, body in _kernels() if "begin_after_previous();" in body}
    assert {"step_kernel", "phi_kernel", "fused_flow_kernel", "flow_tma_kernel", "rim_phi_kernel", "two_steps_3d_kernel",
            "two_steps_2d_kernel", "adjoint_step_kernel"} == set(early)
    for name, params in early.items():
        assert "__restrict__" not in params, name

