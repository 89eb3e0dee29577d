"""Comparisons of products and sums of two floats (csrc/pr_two.cuh), compiled
for the host, against exact arithmetic: products that differ in their last
bits, equal ones, both orders, NaN; temp2_add within 2^-46 of the exact sum
(two units of the low part, 24 bits below the high one's 24)."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2312_04830_gb300 import build

SRC = r"""
#include "pr_two.cuh"
extern "C" void less(long n, const float *v, int *o) {
    for (long i = 0; i < n; ++i) o[i] = prk::product_less(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
}
extern "C" void add(long n, const float *v, float *o) {
    for (long i = 0; i < n; ++i) {
        const prk::Temp2 r = prk::temp2_add({v[3 * i], v[3 * i + 1]}, v[3 * i + 2]);
        o[2 * i] = r.h;
        o[2 * i + 1] = r.l;
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("two")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", build.CSRC, "-o",
                    str(d / "t.so"), str(d / "t.cpp")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)


def test_product_less(lib):
    rng = np.random.default_rng(1)
    n = 4000
    v = np.empty((n, 4), dtype=np.float32)
    v[:, 0] = 3.0
    v[:, 1] = rng.uniform(20.0, 80.0, n)                    # a molar cp
    v[:, 3] = rng.uniform(0.002, 0.05, n)                   # a molar mass
    v[:, 2] = v[:, 0].astype(np.float64) * v[:, 1] / v[:, 3]   # the band's edge, to FP32
    v[::3, 2] = np.nextafter(v[::3, 2], np.float32(0))
    v[1::3, 2] = np.nextafter(v[1::3, 2], np.float32(1e9))
    v[:20, 2:] = v[:20, :2]
    o = np.empty(n, dtype=np.int32)
    lib.less(ctypes.c_long(n), ptr(v), ptr(o))
    F = lambda a: Fraction(float(a))
    assert all(bool(r) == (F(a) * F(b) < F(c) * F(d)) for (a, b, c, d), r in zip(v, o))
    bad = np.array([[3, np.nan, 1, 1], [3, 1, np.nan, 1]], dtype=np.float32)
    lib.less(ctypes.c_long(2), ptr(bad), ptr(o))
    assert not o[:2].any()


def test_sum(lib):
    rng = np.random.default_rng(2)
    n = 4000
    v = np.empty((n, 3), dtype=np.float32)
    v[:, 0] = rng.uniform(60.0, 5000.0, n)
    v[:, 1] = v[:, 0] * rng.uniform(-1, 1, n) * 2.0 ** -25
    v[:, 2] = v[:, 0] * rng.uniform(-0.5, 0.5, n) * 10.0 ** rng.uniform(-9, 0, n)
    o = np.empty((n, 2), dtype=np.float32)
    lib.add(ctypes.c_long(n), ptr(v), ptr(o))
    exact = v.astype(np.float64).sum(axis=1)
    assert (np.abs(o.astype(np.float64).sum(axis=1) - exact) <= 2.0 ** -46 * np.abs(exact)).all()
    assert (o[:, 0] == o.astype(np.float64).sum(axis=1).astype(np.float32)).all()
