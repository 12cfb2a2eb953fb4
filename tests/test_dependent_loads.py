"""Kernels that wait for the grid before them (griddepcontrol.wait) read what it may have written with ordinary loads: the read-only
path (__ldg, const __restrict__) promises data that does not change from the kernel's start, which is before the wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_09615_b200", "csrc")
# weights that are complete before slim_quant's first launch, which is no dependent one
COMPLETE = {"W", "W4"}


def kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__[^{;]*?(\w+)\s*\(([^{;]*)\)\s*\{", text):
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        yield m.group(1), m.group(2), text[m.end():at]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_no_read_only_loads_behind_the_wait(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for kernel, params, body in kernels(text):
        if "after_previous_grid" not in body and "griddepcontrol.wait" not in body:
            continue
        for p in re.findall(r"const[^,]*__restrict__\s*(\w+)", params):
            assert p in COMPLETE, f"{kernel}: {p} is read through the read-only path"
        for arg in re.findall(r"__ldg\(([^;]*)", body):
            assert any(re.search(rf"\b{c}\b", arg) for c in COMPLETE), f"{kernel}: __ldg({arg}"
