"""Which kernels let the next programmatic launch on the stream start before
they have completed: those of the cycle calls, for which the header states what
a caller's kernel must wait for, and those that a later kernel of the same call
follows.
"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2004_02003_gb300", "csrc")


def _kernels_with(text, what):
    """Names of the __global__ functions of a translation unit whose body holds `what`."""
    heads = [(m.start(), m.group(1))
             for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s+)?(\w+)\s*\(", text)]
    return {[name for at, name in heads if at < m.start()][-1] for m in re.finditer(re.escape(what), text)}


def test_only_the_cycle_kernels_launch_dependents_early():
    early = set()
    for src in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        text = re.sub(r"//[^\n]*", "", open(src).read())
        early |= _kernels_with(text, "griddepcontrol.launch_dependents")
    within_a_call = {"fill_copy_kernel", "fill_list_kernel", "fill_interior_kernel"}     # fill_boundary_kernel ends the call
    assert early == {"advect_kernel", "advect_tiled_kernel"} | within_a_call, early
    header = open(os.path.join(ROOT, "include", "bto.h")).read()
    assert "The cycle's kernel (here and in bto_batch_advect_cycle) is launched with" in header
