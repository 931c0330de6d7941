"""The initial-data sweep's quotient (csrc/quotient.cuh), compiled for the host, against exact quotients: within an
ulp over the exponents it is stated for, signs and zeros included, and not finite where an operand is not."""
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
#include "quotient.cuh"
extern "C" void quotients(long n, const double *a, const double *b, double *q) {
  for (long i = 0; i < n; ++i) q[i] = ccz4::quotient(a[i], b[i]);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("quotient")
    src, out = str(d / "quotient.cu"), str(d / "libquotient.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off", "-shared", "-I" + os.path.join(
        ROOT, "paper_2406_11626_gb300", "csrc"), src, "-o", out], check=True, capture_output=True)
    lib = ctypes.CDLL(out)

    def call(a, b):
        a, b = (np.ascontiguousarray(x, dtype=np.float64) for x in np.broadcast_arrays(a, b))
        q, dp = np.empty(a.shape), ctypes.POINTER(ctypes.c_double)
        lib.quotients(ctypes.c_long(a.size), *(x.ctypes.data_as(dp) for x in (a, b, q)))
        return q
    return call


def _check(a, b, q):
    for x, y, z in zip(a, b, q):
        exact = Fraction(x) / Fraction(y)
        # an ulp of the exact quotient's binade
        ulp = Fraction(2) ** (int(np.frexp(float(exact))[1]) - 53)
        assert abs(Fraction(z) - exact) <= ulp, (x, y, z)


@pytest.mark.parametrize("den_exp,num_exp", [((-2, 3), (-2, 3)), ((-60, 60), (-60, 60)), ((-1000, -900), (-60, 20)),
                                             ((900, 1021), (40, 1000)), ((0, 1), (-940, -900)), ((-300, 300), (-300, 300))])
def test_within_an_ulp(run, den_exp, num_exp):
    r = np.random.default_rng(abs(den_exp[0]) + abs(num_exp[1]))
    n = 4000
    b = r.uniform(1.0, 2.0, n) * 2.0 ** r.integers(*den_exp, n) * r.choice([-1.0, 1.0], n)
    a = r.uniform(1.0, 2.0, n) * 2.0 ** r.integers(*num_exp, n) * r.choice([-1.0, 1.0], n)
    keep = (np.abs(np.log2(np.abs(a)) - np.log2(np.abs(b))) < 1020)
    a, b = a[keep], b[keep]
    assert len(a) > 1000
    _check(a, b, run(a, b))


def test_mantissas_at_their_ends(run):
    ends = np.array([1.0, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -23, 1.0 + 2.0 ** -23 - 2.0 ** -52, 1.5, 2.0 - 2.0 ** -52,
                     2.0 - 2.0 ** -23, 2.0 - 2.0 ** -22])
    a, b = (x.reshape(-1) for x in np.meshgrid(ends, ends))
    for s in (1.0, 2.0 ** -700, 2.0 ** 1021):
        q = run(a, b * s) if s < 2.0 ** 1000 else run(a * 2.0 ** 500, b * s)
        _check(a if s < 2.0 ** 1000 else a * 2.0 ** 500, b * s, q)


def test_zeros_and_what_is_not_finite(run):
    assert np.all(run([0.0, -0.0, 0.0], [3.0, 7.0, -1e-200]) == 0.0)
    assert not np.any(np.isfinite(run([1.0, 0.0, np.inf, 5.0, np.nan], [np.inf, -np.inf, np.inf, np.nan, 2.0])))
