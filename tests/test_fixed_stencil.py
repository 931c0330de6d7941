"""The integer stencil sums (csrc/fixed_stencil.cuh), evaluated on the host:
each is the correctly rounded value of the exact sum of its inputs while
they lie within a factor of four (within a few units of 2^-52 of the largest
one otherwise), over the whole range of exponents, and values near or beyond
the top of the FP64 range, infinities and NaN give what FP64 gives."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include <math.h>
#include "fixed_stencil.cuh"
using namespace ccz4;
extern "C" void sums(long n, const double *v, double *out) {
  for (long i = 0; i < n; ++i, v += 19, out += 7) {
    double p[3][3], m[3][3];
    for (int k = 0; k < 3; ++k)
      for (int j = 0; j < 3; ++j) {
        p[k][j] = v[1 + 6 * k + 2 * j];
        m[k][j] = v[2 + 6 * k + 2 * j];
      }
    fx_axes<true, true>(v[0], p, m, out, out + 4, out[3]);
    const double f = fx_first(p[0][0], m[0][0], p[0][1], m[0][1]);
    (void)f;
  }
}
extern "C" double first(double a1, double b1, double a2, double b2) { return fx_first(a1, b1, a2, b2); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("fixed")
    src, out = str(d / "fixed.cu"), str(d / "libfixed.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off", "-shared", "-I" + os.path.join(
        ROOT, "paper_2406_11626_gb300", "csrc"), src, "-o", out], check=True, capture_output=True)
    L = ctypes.CDLL(out)
    L.first.restype = ctypes.c_double
    L.first.argtypes = [ctypes.c_double] * 4
    return L


def _run(lib, v):
    v = np.ascontiguousarray(v, dtype=np.float64)
    out = np.empty((len(v), 7))
    dp = ctypes.POINTER(ctypes.c_double)
    lib.sums(ctypes.c_long(len(v)), v.ctypes.data_as(dp), out.ctypes.data_as(dp))
    return out


def _weights():
    W = np.zeros((7, 19), dtype=int)
    for k in range(3):
        a = 1 + 6 * k
        W[k, [a, a + 1, a + 2, a + 3]] = 8, -8, -1, 1
        W[4 + k, [a, a + 1, a + 2, a + 3, 0]] = 16, 16, -1, -1, -30
        W[3, [a, a + 1, a + 2, a + 3, a + 4, a + 5]] = 15, 15, -6, -6, 1, 1
    W[3, 0] = -60
    return W


@pytest.mark.parametrize("scale", [0, -280, 290, 60])
@pytest.mark.parametrize("spread", [0, 1, 30, 80])
def test_sums_against_exact_rationals(lib, scale, spread):
    r = np.random.default_rng(scale + 7 * spread + 1000)
    v = r.uniform(1.0, 2.0, (200, 19)) * 2.0 ** -r.integers(0, spread + 1, (200, 19)).astype(float)
    if spread:
        v *= r.choice([-1.0, 1.0], v.shape)
    v *= 10.0 ** scale
    v[:20, 3] = 0.0
    v[0] = 0.0
    out, W = _run(lib, v), _weights()
    for i in range(len(v)):
        exact = [sum((int(w) * Fraction(x) for w, x in zip(row, v[i]) if w), Fraction(0)) for row in W]
        top = max(abs(Fraction(x)) for x in v[i])
        for q in range(7):
            err = abs(Fraction(out[i, q]) - exact[q])
            if spread <= 1:  # no bit is dropped: the nearest FP64 number (2^-53 of the result)
                assert err <= abs(exact[q]) * Fraction(1, 2 ** 53), (i, q)
            else:  # dropped bits: one unit of 2^-55 (first) or 2^-53 (others) of the largest value per weight
                unit = top * (Fraction(1, 2 ** 55) if q < 3 else Fraction(1, 2 ** 53))
                assert err <= abs(exact[q]) * Fraction(1, 2 ** 53) + unit * int(np.abs(W[q]).sum()), (i, q)


def test_values_outside_the_integer_range_give_what_fp64_gives(lib):
    with np.errstate(all="ignore"):
        for bad in (np.inf, -np.inf, np.nan, 1e305, -1.7e308):
            for at in (0, 1, 4, 5, 18):
                v = np.linspace(1.0, 2.0, 19)[None].copy()
                v[0, at] = bad
                out = _run(lib, v)[0]
                W = _weights().astype(float)
                ref = np.array([sum(w * x for w, x in zip(row, v[0]) if w) for row in W])
                assert np.array_equal(np.isnan(out), np.isnan(ref)), (bad, at)
                fin = np.isfinite(ref)
                assert np.array_equal(np.isfinite(out), fin) and np.allclose(out[fin], ref[fin], rtol=1e-14)


def test_tiny_and_zero_values(lib):
    v = np.zeros((3, 19))
    v[2, ::2] = -0.0
    assert np.all(_run(lib, v) == 0.0)
    assert lib.first(1e-290, 0.0, 0.0, 0.0) == 8e-290 and lib.first(0.0, 3e-310, 0.0, 0.0) == -8 * 3e-310
    v[1, 1], v[1, 2] = 1e-300, 3e-308
    assert _run(lib, v)[1, 0] == pytest.approx(8 * (1e-300 - 3e-308), rel=1e-15)
