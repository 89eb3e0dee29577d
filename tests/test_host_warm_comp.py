"""The FP32 composition of the FP64 inversion's warm start (csrc/pr_warm.cuh),
compiled for the host, against extended precision.  Bounds: FP32's unit
roundoff (2^-24 of the value; the products with powers of two are exact), plus
the fixed-point steps: each mass fraction short by at most 2^-31, constants off
by 2^-33 of their unit, two units of 2^-31 of a mole fraction, 2^-31 of the
reciprocal.  (From mass fractions rounded to FP32 first: up to 5.8 x 2^-24.)"""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2312_04830_gb300 import build, workloads as W

SRC = r"""
#include <stdint.h>
#include "pr_warm.cuh"
struct C { float x[9], Wbar, bm; };
extern "C" int run(int N, const double *iW, const double *b, long n, const double *Y, float *out) {
    long double w[9], c[9];
    for (int k = 0; k < N; ++k) { w[k] = iW[k]; c[k] = b[k]; }
    prk::WarmTab t;
    if (!prk::fill_warm(t, w, c, N)) return 0;
    for (long i = 0; i < n; ++i) {
        double y[9];
        for (int k = 0; k < 9; ++k) y[k] = k < N ? Y[k * n + i] : 0.0;
        C r;
        prk::warm_comp(t, y, r);
        for (int k = 0; k < 9; ++k) out[11 * i + k] = r.x[k];
        out[11 * i + 9] = r.Wbar;
        out[11 * i + 10] = r.bm;
    }
    return 1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("warm")
    (d / "w.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(d / "w.so"),
                    str(d / "w.cpp")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


def _run(lib, iW, b, Y):
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    Y = np.ascontiguousarray(Y)
    out = np.empty((Y.shape[1], 11), dtype=np.float32)
    assert lib.run(len(iW), ptr(np.ascontiguousarray(iW)), ptr(np.ascontiguousarray(b)), ctypes.c_long(Y.shape[1]), ptr(Y),
                   ptr(out)) == 1
    return out.T


@pytest.mark.parametrize("n_species,kind", [(9, "dirichlet"), (9, "alone"), (9, "trace"), (5, "dirichlet"), (1, "alone")])
def test_against_extended_precision(lib, n_species, kind):
    sp = W.species_table().subset(W.SPECIES[:n_species])
    iW, b = 1.0 / (sp.W * 1e-3), 0.0777960739038885 * 8.314462618 * sp.Tc / sp.pc
    rng = np.random.default_rng(n_species)
    n = 20000
    if kind == "dirichlet":
        Y = W.dirichlet_half(rng, n_species, n)
    elif kind == "alone":
        Y = np.zeros((n_species, n))
        Y[np.arange(n) % n_species, np.arange(n)] = 1.0 + rng.integers(-4000, 4000, n) * 2.0 ** -52
    else:
        Y = 10.0 ** rng.uniform(-14, -1, (n_species, n))
        Y /= Y.sum(axis=0)
    o = _run(lib, iW, b, Y)
    ld = np.longdouble
    m = Y.astype(ld) * iW.astype(ld)[:, None]
    S = m.sum(axis=0)
    x = m / S
    u = ld(2.0) ** -31
    short = u * (iW.astype(ld)[:, None] + x * iW.astype(ld).sum()) / S          # mass fractions
    top = ld(2.0) ** int(np.ceil(np.log2(iW.max())))
    const = ld(2.0) ** -33 * top / iW.astype(ld).min()                         # relative, of 1/W_k
    ex = 2.0 ** -24 * x + short + 2 * u + 2 * const * x
    assert (np.abs(o[:n_species] - x) <= ex).all()
    eW = 2.0 ** -24 + u * iW.sum() / S + const + u
    assert (np.abs(o[9] * S - 1) <= eW).all()
    bm = (x * b.astype(ld)[:, None]).sum(axis=0)
    eb = 2.0 ** -24 + (((short + 2 * u + 2 * const * x) * b.astype(ld)[:, None]).sum(axis=0) / bm) + ld(2.0) ** -31
    assert (np.abs(o[10] / bm - 1) <= eb).all()


def test_refused_mass_fractions_end(lib):
    """NaN, infinities, negative and large values, none at all: any result, no trap."""
    Y = np.array([[np.nan, np.inf, -np.inf, -1.0, 1e300, 2.0, 0.0, -0.0, 5e-324]]).repeat(9, axis=0)
    sp = W.species_table()
    _run(lib, 1.0 / (sp.W * 1e-3), sp.Tc / sp.pc, Y)
