"""The quotients of the plan's factors (csrc/recip.h): a product by the reciprocal corrected by its
remainder, restated in exact rational arithmetic, rounds as a division does."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from conftest import ROOT


def quotient(a, d):
    r = 1.0 / d
    q = a * r
    rem = float(Fraction(a) - Fraction(q) * Fraction(d))          # fma(-q, d, a)
    return float(Fraction(rem) * Fraction(r) + Fraction(q))       # fma(rem, r, q)


@pytest.mark.parametrize("spread", [0, 40, 600])
def test_corrected_quotient_is_the_rounded_one(spread):
    g = np.random.default_rng(spread)
    a = g.standard_normal(4000) * 2.0 ** g.integers(-spread, spread + 1, 4000)
    d = g.uniform(1.0, 2.0, 4000) * 2.0 ** g.integers(-spread // 2, spread // 2 + 1, 4000)
    for x, y in zip(a, d):
        assert quotient(float(x), float(y)) == float(x) / float(y)


SHIM = r"""
#include <cmath>
#include <cstring>
#include <cuda_runtime.h>
static inline int __double2hiint(double x) { long long b; std::memcpy(&b, &x, 8); return (int)(b >> 32); }
using std::fma;
#include "recip.h"
extern "C" void quotients(const double *a, const double *d, double *q, int n) {
  for (int i = 0; i < n; ++i) q[i] = rexi::Recip(d[i]).of(a[i]);
}
extern "C" void complex_quotients(const double2 *a, const double2 *b, double2 *q, int n) {
  for (int i = 0; i < n; ++i) q[i] = rexi::ComplexRecip(b[i]).of(a[i]);
}
"""


@pytest.fixture(scope="module")
def header(tmp_path_factory):
    """csrc/recip.h itself, compiled for the host (every operation in it is IEEE there and on the device)."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    where = tmp_path_factory.mktemp("recip")
    (where / "shim.cpp").write_text(SHIM)
    csrc = os.path.join(ROOT, "paper_1812_03431_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-I", csrc, "-I",
                    os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include"),
                    str(where / "shim.cpp"), "-o", str(where / "shim.so")], check=True)
    lib = ctypes.CDLL(str(where / "shim.so"))

    def run(fn, a, d):
        a, d = np.broadcast_arrays(np.asarray(a), np.asarray(d))
        a, d = np.ascontiguousarray(a), np.ascontiguousarray(d)
        q = np.empty_like(a)
        p = ctypes.c_void_p
        getattr(lib, fn)(p(a.ctypes.data), p(d.ctypes.data), p(q.ctypes.data), a.size)
        return q
    return run


def test_header_rounds_as_the_division(header):
    """Over the whole range of binary64: quotients that over- or underflow, zeros, values that are not
    finite, and both sides of the exponents past which the header divides."""
    g = np.random.default_rng(5)
    edge = [e + k for e in (200 - 1023, 1800 - 1023) for k in (-1, 0, 1)]
    exps = np.array(sorted(set(range(-1022, 1024, 31)) | set(edge) | {-1022, 1023}))
    a, d = (np.ldexp(1.0 + g.random((2, exps.size, exps.size)), np.stack(np.meshgrid(exps, exps, indexing="ij"))))
    a *= g.choice([-1.0, 1.0], a.shape)
    d *= g.choice([-1.0, 1.0], d.shape)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1.0, -3.0])
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(header("quotients", a.ravel(), d.ravel()), (a / d).ravel())
        np.testing.assert_array_equal(header("quotients", special, special[:, None]), special / special[:, None])


def test_header_divides_complex_numbers(header):
    g = np.random.default_rng(6)
    a, b = (g.standard_normal((2, 500)) + 1j * g.standard_normal((2, 500))) * 2.0 ** g.integers(-30, 31, (2, 500))
    q = header("complex_quotients", a, b)
    d = b.real * b.real + b.imag * b.imag
    np.testing.assert_array_equal(q.real, (a.real * b.real + a.imag * b.imag) / d)
    np.testing.assert_array_equal(q.imag, (a.imag * b.real - a.real * b.imag) / d)
