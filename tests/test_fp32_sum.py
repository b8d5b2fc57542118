"""The block sums of FP32 dot partials (csrc/fp32_sum.h), compiled for the host:
never further from the exact sum than additions in FP64, and the same values as
those where FP32 could overflow."""

import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_05930_gb300", "csrc")
SOURCE = """#include "fp32_sum.h"
extern "C" double sum_of(const float* x, int first, int step, int count) { return amgsym::fp32_sum(x, first, step, count); }
"""


@pytest.fixture(scope="module")
def sum_of(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp32_sum")
    (d / "s.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "s.cpp"), "-o", str(d / "s.so")],
                   check=True)
    lib = ctypes.CDLL(str(d / "s.so"))
    lib.sum_of.restype = ctypes.c_double
    lib.sum_of.argtypes = [np.ctypeslib.ndpointer(np.float32), ctypes.c_int, ctypes.c_int, ctypes.c_int]
    return lambda x, first=0, step=1: lib.sum_of(np.ascontiguousarray(x, np.float32), first, step, len(x))


def _inputs(n):
    rng = np.random.default_rng(n)
    yield np.r_[1.0, rng.uniform(0.6, 0.99, n - 1) * 2.0 ** -24]      # every term below half an ulp of the sum
    yield np.r_[rng.uniform(0.6, 0.99, n - 1) * 2.0 ** -24, 1.0]
    yield rng.uniform(0.0, 1.0, n) ** 2                                # <y, y>
    yield rng.standard_normal(n) * 10.0 ** rng.uniform(-20, 20, n)     # spread, both signs
    yield np.r_[rng.standard_normal(n // 2), -rng.standard_normal(n - n // 2)] * 1e-38  # subnormals among them
    x = rng.standard_normal(n).astype(np.float32)
    x[-1] = -np.float32(math.fsum(x[:-1].tolist()))                    # cancels
    yield x


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 9, 15, 16])
def test_no_further_off_than_fp64_additions(sum_of, n):
    for x in _inputs(n):
        x = x.astype(np.float32)
        exact, mag = math.fsum(x.tolist()), math.fsum(np.abs(x).tolist())
        # two roundings of value(), each at most 2^-53 of a result within 2^-24 of the sum, and lo's 2^-61 S
        assert abs(sum_of(x) - exact) <= 2.0 ** -53 * 1.001 * abs(exact) + 2.0 ** -60 * mag


def test_strided(sum_of):
    x = np.random.default_rng(5).standard_normal(85).astype(np.float32)
    for first in range(10):
        assert sum_of(x, first, 10) == pytest.approx(math.fsum(x[first::10].tolist()), rel=1e-14)


def test_what_fp32_could_not_hold(sum_of):
    f = np.float32
    assert sum_of([2e38, 2e38, 2e38, -2e38]) == float(f(2e38)) * 2       # FP32 would overflow on the way
    assert sum_of([f(2e38)] * 16) == float(f(2e38)) * 16
    assert sum_of([1.0, np.inf, 2.0]) == np.inf and sum_of([1.0, -np.inf]) == -np.inf
    assert math.isnan(sum_of([np.inf, -np.inf])) and math.isnan(sum_of([1.0, np.nan, 2.0]))
    assert sum_of([2.0 ** 89] * 16) == 2.0 ** 93 and sum_of([]) == 0.0
