"""Kernels that wait for the grid before them may be in flight while it still writes what they read,
so they must not read it as data that is constant for their lifetime: no __ldg, no const __restrict__
input.  Checked in the source; no GPU."""
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2405_03605_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_dependent_kernels_read_no_constant_data():
    seen = 0
    for name in ("ga_mrca.cu", "ga_async.cu", "ga_step.cu", "ga_resident.cu"):
        for kernel in re.split(r"(?=__global__)", source(name))[1:]:
            # a kernel whose grid may be launched before the one it depends on has ended
            if "wait_previous_grid" not in kernel.split("\n}\n")[0]:
                continue
            seen += 1
            head = kernel[:kernel.index("\n}\n")]
            assert "__ldg" not in head, head[:120]
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", head), head[:200]
    assert seen >= 9
    # the bodies that the step kernels share, and their parameters
    body = source("ga_island.cuh")
    assert "__ldg" not in body
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", body)
    assert "__ldg" not in source("ga_mrca.cu")
