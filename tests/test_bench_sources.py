"""The profiled traffic of bench.py is tied to every file that decides it: the
kernels of the solve step, what they include, and the tile choice."""

import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2407_05930_gb300", "csrc")


def test_profiled_traffic_names_the_files_it_depends_on():
    named = {os.path.basename(f) for f in bench.KERNEL_SOURCES}
    todo, seen = ["k_spmm.cu", "k_misc.cu"], set()
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        todo += re.findall(r'#include "(\w+\.\w+)"', open(os.path.join(CSRC, f)).read())
    seen -= {"internal.h"}  # host types and the C interface's includes
    assert seen | {"solve.cu"} <= named
    assert "fixed_tile(" in open(os.path.join(CSRC, "solve.cu")).read()
    assert all(os.path.exists(os.path.join(bench.ROOT, f)) for f in bench.KERNEL_SOURCES)
