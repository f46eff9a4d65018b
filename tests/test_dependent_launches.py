"""Kernels launched as programmatic dependents start while the kernel before
them still writes: they wait (griddepcontrol.wait) and read afterwards.  A
``__restrict__`` pointer among their parameters would tell the compiler that
nobody else writes that memory while they run, and allow loads ahead of the
wait and through the read-only cache.  Read off the sources: no GPU."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WAIT = ("griddepcontrol.wait", "pdl_wait_and_release();")


def dependent_kernels():
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_1412_5170_gb300", "csrc", "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void[^;{]*?\b(k_\w+)\(([^{;]*)\)\s*\{(.*?)\n\}", text, re.S):
            if any(w in m.group(3) for w in WAIT):
                yield os.path.basename(path), m.group(1), m.group(2)


KERNELS = list(dependent_kernels())


def test_the_dependent_kernels_are_found():
    names = {k for _, k, _ in KERNELS}
    assert {"k_step_generic", "k_step_walk", "k_step_strip", "k_step_batch_tiles", "k_step_batch_walk", "k_net",
            "k_net_grad"} <= names


@pytest.mark.parametrize("path,name,params", KERNELS, ids=[k for _, k, _ in KERNELS])
def test_no_restrict_parameter(path, name, params):
    assert "__restrict__" not in params, (path, name)
