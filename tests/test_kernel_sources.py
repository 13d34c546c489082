"""Rules that the compiler does not check, read off the kernels' sources."""
import os
import re

import pytest

from paper_2506_02114_gb300 import build

# copied to the device before a plan's first kernel, written by no kernel
INPUTS = {"pos", "m", "MMop", "MLop", "LLop", "inv"}


def early_kernels():
    """(file, kernel, parameters) of the kernels that may be set up while the
    stream's kernel before them still runs (grid_begin)."""
    for src in build.SOURCES:
        with open(os.path.join(build.CSRC, src)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(([^{]*)\)\s*\{\s*"
                             r"grid_begin\(\);", text):
            yield src, m.group(1), m.group(2)


def test_the_early_kernels_are_found():
    names = {k for _, k, _ in early_kernels()}
    assert {"k_gather_stars", "k_tree_top", "k_p2m", "k_m2m", "k_local", "k_leaf_finalize"} <= names


@pytest.mark.parametrize("src,kernel,params", list(early_kernels()),
                         ids=lambda v: v if v.startswith("k_") else "")
def test_no_promise_of_constancy_for_what_an_earlier_kernel_writes(src, kernel, params):
    """`const T *__restrict__` promises that nothing writes the data while the
    kernel runs, and lets its loads move ahead of the wait in grid_begin."""
    promised = {m.group(1) for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params)}
    assert promised <= INPUTS, "%s: %s" % (src, sorted(promised - INPUTS))
