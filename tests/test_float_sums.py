"""The FP32 sums of the kernels (csrc/compensated.h), compiled for the host with g++."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from helpers import ROOT

SRC = r"""
#include "compensated.h"
extern "C" float joined(const float* x, int n) {
    float total = 0.f, low = 0.f;
    for (int i = 0; i < n; ++i) stdg::join(total, low, x[i]);
    return total + stdg::rest(total, low);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("sums")
    (d / "sums.cpp").write_text(SRC)
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1802_04516_gb300", "csrc"), "-o", str(d / "sums.so"), str(d / "sums.cpp")], check=True)
    out = ctypes.CDLL(str(d / "sums.so"))
    out.joined.restype = ctypes.c_float
    out.joined.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return out


@pytest.mark.parametrize("n", [1, 2, 5, 64, 1000])
def test_joined_sum_is_the_rounded_sum_while_the_total_is_the_larger(lib, n):
    # with |total| >= |term| at every join the collected errors are exact to first order: within one unit in the last
    # place of the result plus n^2 eps^2 of the sum of the magnitudes
    rng = np.random.default_rng(n)
    for _ in range(20):
        x = np.sort(rng.uniform(0.1, 1.0, n).astype(np.float32))[::-1].copy()
        exact = float(sum(Fraction(float(v)) for v in x))
        got = lib.joined(x.ctypes.data, n)
        assert abs(got - exact) <= 2.0 ** -24 * exact + (n * 2.0 ** -24) ** 2 * exact


def test_infinite_total_stays_infinite(lib):
    for x, want in (([1.0, np.inf, 2.0], np.inf), ([-np.inf, 1e30], -np.inf), ([3e38, 3e38, -1e38], np.inf)):
        x = np.array(x, dtype=np.float32)
        assert lib.joined(x.ctypes.data, x.size) == want
    x = np.array([np.inf, -np.inf, 1.0], dtype=np.float32)
    assert np.isnan(lib.joined(x.ctypes.data, 3))
