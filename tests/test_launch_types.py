"""Kernel launches are type-checked by the compiler: pointers of another type,
dropped const and swapped arguments do not compile (csrc/pdl.cuh)."""

import os
import subprocess

import pytest

import paper_2407_05930_gb300.build as build

SOURCE = """#include "pdl.cuh"
namespace amgsym { thread_local PdlState t_pdl; }
__global__ void kern(const float* a, double* b, int64_t n) {}
void launch(float* f, double* d, const double* cd, int n) {
  amgsym::launch_pdl(kern, 1, 32, 0, (cudaStream_t)0, %s);
}
"""


@pytest.mark.parametrize("args,ok", [("f, d, n", True), ("nullptr, d, 5", True), ("d, d, n", False), ("f, cd, n", False),
                                     ("d, f, n", False), ("f, d", False)])
def test_launch_arguments(tmp_path, args, ok):
    src = tmp_path / "launch.cu"
    src.write_text(SOURCE % args)
    r = subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-c", str(src), "-o",
                        os.fspath(tmp_path / "launch.o")], capture_output=True, text=True)
    assert (r.returncode == 0) == ok, r.stderr
