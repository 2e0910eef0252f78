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
template <int CH> static float row(const float* k, const float* x, int slots, int n) {
    stdg::RowSum<float> r;
    for (int s = 0; s < slots; ++s) {
        for (int c = 0; c < n; c += CH) {
            float kv[CH];
            for (int j = 0; j < CH; ++j) kv[j] = k[s * n + c + j];
            r.columns(kv, [&](int j) { return x[s * n + c + j]; });
        }
        r.end_slot();
    }
    return r.scaled(1.f);
}
extern "C" float row_sum(const float* k, const float* x, int slots, int n) {
    return n % 10 == 0 ? row<10>(k, x, slots, n) : row<6>(k, x, slots, n);
}
extern "C" double tree(const float* s, const float* c) {   // 32 lanes, as the butterfly adds them in lane 0
    stdg::Triple v[32];
    for (int i = 0; i < 32; ++i) v[i] = stdg::Triple{s[i], c[i], 0.f};
    for (int o = 16; o > 0; o >>= 1)
        for (int i = 0; i < o; ++i) v[i].plus(v[i + o]);
    return v[0].value();
}
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
    out.row_sum.restype = ctypes.c_float
    out.row_sum.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    out.tree.restype = ctypes.c_double
    out.tree.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
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


@pytest.mark.parametrize("slots,n", [(4, 6), (4, 12), (4, 30), (5, 12), (5, 60)])
def test_row_sum_of_conjugate_gradients(lib, slots, n):
    # the operator row inside the fused CG kernels: root mean square error over random rows at most 0.9 of that of plain
    # FP32 totals of chains of 10 or 6 products (0.7 to 0.85 expected; 1 without the compensation)
    rng = np.random.default_rng(n)
    rows, ch = 4000, 10 if n % 10 == 0 else 6
    K, X = rng.normal(size=(2, rows, slots * n)).astype(np.float32)
    exact = np.sum(K.astype(np.float64) * X, axis=1)
    got = np.array([lib.row_sum(k.ctypes.data, x.ctypes.data, slots, n) for k, x in zip(K, X)], dtype=np.float64)
    total = np.zeros(rows, dtype=np.float32)
    for s in range(slots):
        slot = np.zeros(rows, dtype=np.float32)
        for c in range(s * n, (s + 1) * n, ch):
            chain = np.zeros(rows, dtype=np.float32)
            for j in range(c, c + ch):
                chain = (K[:, j].astype(np.float64) * X[:, j] + chain).astype(np.float32)
            slot += chain
        total += slot
    rms = lambda e: np.sqrt(np.mean(e ** 2))  # noqa: E731
    assert rms(got - exact) < 0.9 * rms(total.astype(np.float64) - exact)


@pytest.mark.parametrize("cancel", [False, True])
@pytest.mark.parametrize("scale", [1.0, 1e30, 1e-30])
def test_lane_tree_loses_no_bit_of_fp64(lib, cancel, scale):
    # FP32 inner products reach the tree over the lanes as pairs s + c, |c| some 2^-24 |s|. Its result is the exact sum
    # rounded to FP64, up to 2^-68 of the magnitudes (six additions of third terms at 2^-24 of 2^-48 each, with room) and
    # the smallest subnormal
    rng = np.random.default_rng(5)
    for _ in range(200):
        s = (scale * rng.normal(size=32) * 2.0 ** rng.integers(-6, 7, 32)).astype(np.float32)
        if cancel:
            s[16:] = -s[:16]
        c = (s * 2.0 ** -24 * rng.uniform(-8, 8, 32)).astype(np.float32)
        exact = sum(Fraction(float(v)) for v in s) + sum(Fraction(float(v)) for v in c)
        got = Fraction(lib.tree(s.ctypes.data, c.ctypes.data))
        mag = sum(abs(Fraction(float(v))) for v in s)
        assert abs(got - exact) <= abs(exact) * Fraction(2) ** -52 + mag * Fraction(2) ** -68 + 64 * Fraction(2) ** -149
