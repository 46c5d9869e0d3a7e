"""The three-float sums of the cluster statistics are no less accurate than the FP64 sums they stand for: the header compiled
for the host, against exact sums (products of two floats are exact in double, math.fsum adds them exactly)."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_02010_gb300", "csrc")
SRC = r"""
#include "threefloat.cuh"
extern "C" double dot(const float *a, const float *b, int n, int *exact) {
    otgb::ThreeFloat s;
    for (int i = 0; i < n; ++i) s.add_product(a[i], b[i]);
    *exact = s.exact;
    return s.value();
}
"""


@pytest.fixture(scope="module")
def dot(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("tf")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-x", "c++", "-I", CSRC, str(d / "t.cpp"),
                    "-o", str(d / "t.so")], check=True)
    f = ctypes.CDLL(str(d / "t.so")).dot
    f.restype = ctypes.c_double
    p = ctypes.POINTER(ctypes.c_float)

    def call(a, b):
        e = ctypes.c_int()
        a, b = (np.ascontiguousarray(v, np.float32) for v in (a, b))
        return f(a.ctypes.data_as(p), b.ctypes.data_as(p), len(a), ctypes.byref(e)), bool(e.value)

    return call


@pytest.mark.parametrize("kind", ["plain", "cancel", "wide", "offset"])
def test_no_less_accurate_than_double(dot, kind):
    rng = np.random.default_rng(3)
    n = 20_000
    a = rng.uniform(0.5, 1.5, n).astype(np.float32)
    b = {"plain": rng.normal(size=n), "cancel": np.repeat(rng.normal(size=n // 2) * 1e6, 2) * np.tile([1.0, -1.0], n // 2),
         "wide": rng.normal(size=n) * 10.0 ** rng.integers(-6, 7, n), "offset": 1e5 + rng.normal(size=n)}[kind].astype(np.float32)
    if kind == "cancel":
        a = np.repeat(a[::2], 2)
        b[-1] = 1.0
    got, exact = dot(a, b)
    prod = a.astype(np.float64) * b.astype(np.float64)
    want = math.fsum(prod)
    plain = 0.0
    for v in prod:
        plain += v
    assert exact
    # one rounding to double, and 2^-60 of the terms; a double sum of n terms is off by up to n 2^-53 of them
    assert abs(got - want) <= 2.0 ** -52 * abs(want) + 2.0 ** -60 * float(np.abs(prod).sum())
    assert abs(got - want) <= abs(plain - want) + 2.0 ** -52 * abs(want)


def test_products_near_the_denormal_range_are_flagged(dot):
    assert dot([1e-20, 1.0], [1e-15, 1.0])[1] is False
    assert dot([0.0, 1.0], [1e-38, 1.0])[1] is True
