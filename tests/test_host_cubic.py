"""The cubic's single root with FP32 seeds and derivatives (csrc/pr_cubic.cuh),
compiled for the host, against 60-digit roots of the same coefficients: from
the critical point (T and p within 1e-13 to 1e-2 of it, where the three roots
meet) to gas and liquid states.  A root it gives is off by at most the FP64
residual's rounding over the derivative: four roundings of at most the terms'
magnitudes, twice over for the step that follows (8 x 2^-53).  It has to give
one in usual states (at low pressure the two roots near 0 are nearly double,
and their count is left to the general form)."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2312_04830_gb300 import build

mpmath = pytest.importorskip("mpmath")

SRC = r"""
#include <stdint.h>
#include "pr_cubic.cuh"
extern "C" void run(long n, const double *c2, const double *c1, const double *c0, const double *B, double *Z, int *ok) {
    for (long i = 0; i < n; ++i) ok[i] = prk::cubic_single_root(c2[i], c1[i], c0[i], B[i], Z[i]);
}
"""


@pytest.fixture(scope="module")
def single_root(tmp_path_factory):
    d = tmp_path_factory.mktemp("cubic")
    (d / "c.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(d / "c.so"),
                    str(d / "c.cpp")], check=True)
    L = ctypes.CDLL(str(d / "c.so"))

    def call(c2, c1, c0, B):
        a = [np.ascontiguousarray(v, dtype=np.float64) for v in (c2, c1, c0, B)]
        Z, ok = np.zeros(a[0].size), np.zeros(a[0].size, dtype=np.int32)
        L.run(ctypes.c_long(Z.size), *(v.ctypes.data_as(ctypes.c_void_p) for v in (*a, Z, ok)))
        return Z, ok.astype(bool)
    return call


def _cubic(Tr, pr, kappa):
    al = (1.0 + kappa * (1.0 - np.sqrt(Tr))) ** 2
    A, B = 0.457235528921382 * pr / Tr ** 2 * al, 0.0777960739038885 * pr / Tr
    return B - 1.0, A - B * (3.0 * B + 2.0), B * (B + B * B - A), B


def _check(Z, ok, c2, c1, c0):
    mpmath.mp.dps = 60
    worst = 0.0
    for z, b2, b1, b0 in zip(Z[ok], c2[ok], c1[ok], c0[ok]):
        m = mpmath.mpf(float(z))
        b2, b1, b0 = (mpmath.mpf(float(v)) for v in (b2, b1, b0))
        f, g = ((m + b2) * m + b1) * m + b0, (3 * m + 2 * b2) * m + b1
        terms = m ** 3 + abs(b2) * m ** 2 + abs(b1) * m + abs(b0)
        # the distance to the root is |f / f'| to first order where the root is simple
        worst = max(worst, float(abs(f) / (8 * mpmath.mpf(2) ** -53 * terms)))
        assert abs(f * (6 * m + 2 * b2)) < 1e-3 * g * g, (float(f), float(g))   # a simple root's neighbourhood
    return worst


@pytest.mark.parametrize("exponent", [2, 4, 6, 8, 9, 10, 11, 13])
def test_near_the_critical_point(single_root, exponent):
    rng = np.random.default_rng(exponent)
    s = 10.0 ** -exponent
    c2, c1, c0, B = _cubic(1.0 + s * rng.uniform(-1, 1, 400), 1.0 + s * rng.uniform(-1, 1, 400), 0.5)
    Z, ok = single_root(c2, c1, c0, B)
    assert _check(Z, ok, c2, c1, c0) <= 1.0


@pytest.mark.parametrize("Tr,pr,kappa", [((1.2, 20.0), (1.5, 3.0), 0.5), ((1.1, 3.0), (0.5, 3.0), 0.05),
                                         ((0.6, 0.95), (1.5, 4.0), 0.8)])
def test_usual_states(single_root, Tr, pr, kappa):
    rng = np.random.default_rng(7)
    c2, c1, c0, B = _cubic(rng.uniform(*Tr, 400), rng.uniform(*pr, 400), kappa)
    Z, ok = single_root(c2, c1, c0, B)
    assert ok.mean() > 0.95 and _check(Z, ok, c2, c1, c0) <= 1.0
