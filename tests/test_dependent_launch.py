"""Kernels launched before their predecessor has ended (pgb_internal.cuh: launch_dependent) read and
write memory that changes while they run, so __restrict__ -- which promises that it does not -- may
qualify their pointers to the plan's constants only.  Checked on the sources: the fault it would be
(a load moved ahead of grid_wait, or through the non-coherent path) depends on code generation."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_08806_gb300", "csrc")
CONSTANTS = {"A", "D", "E", "scale"}  # transform matrices and node scales, written when the plan is made


def _dependent_kernels():
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for part in text.split("__global__")[1:]:
            head, body = part.split("{", 1)
            if "grid_wait();" in body.split("\n}\n", 1)[0]:
                yield name, re.search(r"\b(k_\w+)\s*\(", head).group(1), head


def test_only_constants_are_restrict_qualified():
    found = {}
    for name, kernel, head in _dependent_kernels():
        found[kernel] = set(re.findall(r"__restrict__\s+(\w+)", head))
    assert {"k_axis_pass_pair", "k_recon_last", "k_loss_mirror", "k_final", "k_spread_f32", "k_spread_f64"} <= set(found)
    assert all(q <= CONSTANTS for q in found.values()), found
