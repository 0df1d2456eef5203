"""The step-size rule's sum of squares (csrc/wide_sum.cuh), compiled for the host and added in the kernel's
order, against exact rational arithmetic: within one FP64 rounding, also where it holds 28,000 entries."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_0908_4421_gb300 import build as cuda_build

HARNESS = """
#include "wide_sum.cuh"
using namespace imrt;
extern "C" double sum_squares(const float* w, int n) {
    WideSum lane[512] = {};
    for (int t = 0; t < 512; ++t)
        for (int i = t; i < n; i += 512) lane[t] = wide_add(lane[t], wide_square(w[i]));
    for (int o = 16; o > 0; o >>= 1) {
        WideSum next[512];
        for (int t = 0; t < 512; ++t) next[t] = wide_add(lane[t], lane[t ^ o]);
        for (int t = 0; t < 512; ++t) lane[t] = next[t];
    }
    WideSum part[16];
    for (int k = 0; k < 16; ++k) part[k] = lane[32 * k];
    for (int o = 8; o > 0; o >>= 1) {
        WideSum next[16];
        for (int k = 0; k < 16; ++k) next[k] = wide_add(part[k], part[k ^ o]);
        for (int k = 0; k < 16; ++k) part[k] = next[k];
    }
    return wide_to_double(part[0]);
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide_sum")
    src, lib = d / "sums.cpp", d / "sums.so"
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-x", "c++", "-I",
                           cuda_build.CSRC, "-o", str(lib), str(src)])
    fn = ctypes.CDLL(str(lib)).sum_squares
    fn.restype = ctypes.c_double
    return fn


@pytest.mark.parametrize("n", [1, 2, 511, 513, 1030, 3140, 28000])
@pytest.mark.parametrize("decades", [0, 3, 12])
def test_sum_of_squares_is_rounded_once(sums, n, decades):
    rng = np.random.Generator(np.random.PCG64(n + decades))
    w = (rng.uniform(0.5, 1.99, n) * 10.0 ** -rng.uniform(0, decades, n)).astype(np.float32)
    exact = sum((Fraction(float(v)) ** 2 for v in w), Fraction(0))
    got = Fraction(sums(w.ctypes.data_as(ctypes.c_void_p), n))
    # what the three floats leave out (about n^2 2^-72) is far below the last rounding
    assert abs(got - exact) <= exact * Fraction(1, 2 ** 53) * (1 + Fraction(1, 1000))
