"""The files behind a kernel decide whether a committed capture is still the kernel's, and whether its layouts
round alike."""
import os
import re

import pytest

import bench
from paper_2404_02521_gb300 import build


def closure(names):
    """The files and every file of the same folder that they include, directly or not."""
    seen, todo = set(), list(names)
    while todo:
        n = todo.pop()
        if n not in seen:
            seen.add(n)
            text = open(os.path.join(build.CSRC, n)).read()
            todo += [i for i in re.findall(r'#include "([^"/]+)"', text) if os.path.exists(os.path.join(build.CSRC, i))]
    return seen


@pytest.mark.parametrize("kernel", sorted(bench.KERNEL_SOURCES))
def test_captures_follow_every_source(kernel):
    listed = {os.path.basename(s) for s in bench.KERNEL_SOURCES[kernel]}
    text = {f: open(os.path.join(build.CSRC, f)).read() for f in os.listdir(build.CSRC) if f.endswith(".cu")}
    # the files that define the kernel or instantiate its definition, and the one that plans its launches
    home = {f for f, t in text.items() if re.search(r"\b%s\(" % kernel, t)}
    if kernel == "fine_tile_kernel":
        home |= {f for f, t in text.items() if "BS_FINE_INSTANCE(" in t} | {"fine.cu"}
    assert listed == closure(home)


def test_layouts_that_agree_bitwise_are_compiled_without_contraction():
    # F's planner and every file that instantiates its tiles, and the grid solver's layouts
    exact = [f for f in os.listdir(build.CSRC) if f.endswith(".cu") and
             ("BS_FINE_INSTANCE(" in open(os.path.join(build.CSRC, f)).read() or f in ("fine.cu", "coarse_grid.cu"))]
    assert len(exact) > 2
    for f in exact + ["fine_wz.cu"]:
        assert "-fmad=false" in build.file_flags(f), f
    for f in ("coarse.cu", "fine3.cu", "pino.cu"):
        assert build.file_flags(f) == [], f
