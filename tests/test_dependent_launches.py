"""Kernels that run while the launch before them still writes (launch_early, fx_after) must not
declare what that launch writes as const __restrict__: the compiler may take such memory for
read-only during the whole kernel and load it ahead of the wait.  A check of the sources."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1810_00900_gb300" / "csrc"
# uploaded before the first launch of a chain and not written by any of its launches
PLAN = {"segs", "trees", "lvl_off"}


def kernels():
    """name -> (parameter list, body) of every __global__ function."""
    found = {}
    for f in sorted(CSRC.glob("*.cu*")):
        src = re.sub(r"//[^\n]*", "", f.read_text())
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^)]*\) )?(\w+)\(([^{};]*)\)\s*\{", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            found[m.group(1)] = (m.group(2), src[m.end():i])
    return found


def launched_early():
    text = "".join(f.read_text() for f in sorted(CSRC.glob("*.cuh")) + sorted(CSRC.glob("*.cu")))
    return set(re.findall(r"launch_early\([^;]*?\b(\w+_kernel)<", text))


def test_kernels_are_found():
    assert {"fx_level_warp_kernel", "fx_level_cta_kernel", "fx_leaf_kernel", "fx_final_kernel"} <= launched_early()
    assert launched_early() <= set(kernels())


@pytest.mark.parametrize("name", sorted(launched_early()))
def test_dependent_kernels_wait_and_qualify_only_the_plan(name):
    params, body = kernels()[name]
    if "fx_after()" in body:
        marked = {re.search(r"(\w+)\s*$", p).group(1) for p in params.split(",") if "__restrict__" in p}
        assert marked <= PLAN
    else:  # reads only what was complete before the launch beside it began; ends after that one
        assert body.index("griddepcontrol.launch_dependents") < body.rindex("griddepcontrol.wait")
        assert body.rstrip("} \n").endswith('asm volatile("griddepcontrol.wait;" ::: "memory");')
