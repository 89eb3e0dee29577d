"""The integer-pipe functions (csrc/pr_int64.cuh), compiled for the host,
against 60-digit arithmetic: reciprocal and inverse square root within 2^-59
relative, 2^-f and log2 within 2^-59 absolute (the bounds the rounded
functions of csrc/pr_math64.cuh rest on: 2^-59 is 1/64 of a unit in the last
place).  The hardware's single-precision reciprocal and inverse square root
are replaced by the host's with up to two units of error either way."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_04830_gb300", "csrc")
SRC = r"""
#include <stdint.h>
#include <math.h>
extern "C" { int seed_error = 0; }
static float bump(float v) { for (int k = 0; k < seed_error; ++k) v = nextafterf(v, 9.f);
                             for (int k = 0; k > seed_error; --k) v = nextafterf(v, 0.f); return v; }
#define HOST_RCP(x) bump(1.0f / (x))
#define HOST_RSQRT(x) bump(1.0f / sqrtf(x))
#include "pr_int64.cuh"
extern "C" void run(int fn, long n, const uint64_t *x, uint64_t *y) {
    for (long i = 0; i < n; ++i)
        y[i] = fn == 0 ? i64::rcp_m(x[i]) : fn == 1 ? i64::rsqrt_m(x[i]) : fn == 2 ? i64::exp2_neg(x[i]) : i64::log2_m(x[i]);
}
"""


@pytest.fixture(scope="module")
def fn(tmp_path_factory):
    d = tmp_path_factory.mktemp("int64")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    L = ctypes.CDLL(str(d / "t.so"))

    def call(which, x, seed=0):
        ctypes.c_int.in_dll(L, "seed_error").value = seed
        x = np.ascontiguousarray(x, dtype=np.uint64)
        y = np.empty_like(x)
        L.run(which, ctypes.c_long(x.size), x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p))
        return [int(v) for v in y]
    return call


def _args(lo, hi, n=400):
    rng = np.random.default_rng(11)
    edges = [lo, lo + 1, lo + 2048, hi - 1, hi - 2, (lo + hi) // 2, (lo + hi) // 2 + 1]
    edges += [lo + (hi - lo) // 1024 * k + d for k in (1, 255, 256, 511, 1000) for d in (-1, 0, 1)]
    return np.array(edges + [lo + int(v) for v in rng.integers(0, hi - lo, n, dtype=np.uint64)], dtype=np.uint64)


@pytest.mark.parametrize("seed", [-2, -1, 0, 1])
@pytest.mark.parametrize("which", [0, 1])
def test_reciprocal_and_inverse_root(fn, which, seed):
    mpmath.mp.dps = 60
    x = _args(1 << 63, 1 << 64) if which == 0 else _args(1 << 62, 1 << 64)
    worst = 0
    for a, r in zip(x, fn(which, x, seed)):
        if which == 0:
            e = mpmath.mpf(r) / 2 ** 64 * mpmath.mpf(int(a)) / 2 ** 63 - 1
        else:
            e = mpmath.mpf(r) / 2 ** 63 * mpmath.sqrt(mpmath.mpf(int(a)) / 2 ** 64) - 1
        worst = max(worst, abs(e))
    assert worst <= mpmath.mpf(2) ** -59


@pytest.mark.parametrize("which", [2, 3])
def test_exp2_and_log2(fn, which):
    mpmath.mp.dps = 60
    x = _args(0, 1 << 64) if which == 2 else _args(1 << 63, 1 << 64)
    worst = 0
    for a, r in zip(x, fn(which, x)):
        a = mpmath.mpf(int(a))
        e = mpmath.mpf(r) / 2 ** 63 - mpmath.power(2, -a / 2 ** 64) if which == 2 else \
            mpmath.mpf(r) / 2 ** 64 - mpmath.log(a / 2 ** 63, 2)
        worst = max(worst, abs(e))
    assert worst <= mpmath.mpf(2) ** -59
