"""The stencil sums of the derivative pass (csrc/fixed_stencil.cuh: words and
exponents, fx_point, fx_first_sum) and the 7-point Laplacian of the initial-data
sweep, compiled for the host and compared with exact rationals: each sum is
correctly rounded while its own values lie within a factor of sixteen of the
largest of them, whatever the values that it does not have, and otherwise off by
at most one unit of 2^-56 of the largest for each unit of weight; f -> -f and a
reflection change the sign of a result and no bit; zeros of either sign add
nothing; and on smooth data that cross zero the error is no larger than that of
the same sums in FP64."""
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
// v: [19] centre, then per axis +1, -1, +2, -2, +3, -3; out: [10] the seven sums, the first sums alone
extern "C" void sums(long n, const double *v, double *out) {
  const int st[3] = {1, 4, 16};
  for (long i = 0; i < n; ++i, v += 19, out += 10) {
    int64_t w[97];
    unsigned short e[97];
    auto put = [&](int at, double x) {
      unsigned q;
      w[48 + at] = fx_word(x, q);
      e[48 + at] = (unsigned short)q;
    };
    put(0, v[0]);
    for (int k = 0; k < 3; ++k)
      for (int j = 0; j < 3; ++j) {
        put((j + 1) * st[k], v[1 + 6 * k + 2 * j]);
        put(-(j + 1) * st[k], v[2 + 6 * k + 2 * j]);
      }
    fx_point<true, false>(w + 48, e + 48, st, out);
    for (int k = 0; k < 3; ++k) out[7 + k] = fx_first_sum(w + 48, e + 48, st[k]);
  }
}
extern "C" void values(long n, const double *v, double *out) {
  for (long i = 0; i < n; ++i) {
    unsigned e;
    const int64_t w = fx_word(v[i], e);
    out[i] = fx_value(w, e);
  }
}
extern "C" void laplacian(long n, const double *v, double *out) {
  for (long i = 0; i < n; ++i, v += 7) out[i] = fx_laplacian(v[0], {v[1], v[2], v[3], v[4], v[5], v[6]});
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("sums")
    src, out = str(d / "sums.cu"), str(d / "libsums.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off", "-shared", "-I" + os.path.join(
        ROOT, "paper_2406_11626_gb300", "csrc"), src, "-o", out], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _call(f, v, width):
    v = np.ascontiguousarray(v, dtype=np.float64)
    out = np.empty((len(v), width))
    dp = ctypes.POINTER(ctypes.c_double)
    f(ctypes.c_long(len(v)), v.ctypes.data_as(dp), out.ctypes.data_as(dp))
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


W = _weights()
OWN = W != 0   # the values that set a sum's unit


def _exact(v):
    return [sum((int(w) * Fraction(x) for w, x in zip(row, v) if w), Fraction(0)) for row in W]


def _exponent(v):
    """floor(log2) of each magnitude; far below every other of zero."""
    return np.where(v == 0.0, -5000, np.frexp(v)[1] - 1)


def _samples(seed, n, spread):
    r = np.random.default_rng(seed)
    v = r.uniform(1.0, 2.0, (n, 19)) * 2.0 ** -r.integers(0, spread + 1, (n, 19)).astype(float)
    return v * r.choice([-1.0, 1.0], v.shape)


@pytest.mark.parametrize("scale", [0, -200, 280])
@pytest.mark.parametrize("spread", [0, 2, 4, 9, 30, 70, 300])
def test_sums_against_exact_rationals(lib, scale, spread):
    v = _samples(scale + 31 * spread + 400, 150, spread)
    v[:30, 3] = 0.0
    v[30:40, 0] = -0.0
    v *= 2.0 ** scale
    out, e = _call(lib.sums, v, 10), _exponent(v)
    for i in range(len(v)):
        ex = _exact(v[i])
        for q in range(7):
            top = int(e[i][OWN[q]].max())
            dropped = (e[i] < top - 4) & (v[i] != 0.0)
            unit = Fraction(2) ** (top - 56)
            # one unit for each unit of weight of a value with dropped bits; where there is one, a second derivative
            # may truncate its neighbours' part once more, the dissipation three axes' parts of weight three and a
            # sum formed in fourths of its unit
            bar = unit * int(np.abs(W[q])[dropped].sum()) if q != 3 or not dropped.any() else unit * (192 + 9 + 4)
            bar += unit if q > 3 and dropped.any() else 0
            bar += abs(ex[q]) * Fraction(1, 2 ** 53)
            got = [out[i, q]] + ([out[i, 7 + q]] if q < 3 else [])
            for g in got:
                assert abs(Fraction(g) - ex[q]) <= bar, (i, q, g, float(ex[q]))


@pytest.mark.parametrize("ratio", [1e-2, 1e-6, 1e-20, 1e-150])
@pytest.mark.parametrize("at", [0, 5, 6, 7, 17])
def test_a_derivative_does_not_lose_bits_to_other_neighbours(lib, ratio, at):
    """Along x within a factor of four, everything else far below one neighbour at distance three or on another axis, or below the centre."""
    r = np.random.default_rng(at)
    v = r.uniform(1.0, 2.0, (100, 19)) * 2.0 ** -r.integers(0, 2, (100, 19)).astype(float) * ratio
    v[:, at] = 1.25
    out = _call(lib.sums, v, 10)
    for i in range(len(v)):
        ex = _exact(v[i])
        for q in (0, 4) if at else (0,):
            assert abs(Fraction(out[i, q]) - ex[q]) <= abs(ex[q]) * Fraction(1, 2 ** 53), (i, q)


@pytest.mark.parametrize("spread", [0, 3, 8, 20, 60, 90, 600])
def test_symmetries_are_exact(lib, spread):
    v = _samples(spread + 7, 400, spread)
    r = np.random.default_rng(spread)
    v[r.random(v.shape) < 0.1] = 0.0
    v[r.random(v.shape) < 0.1] = -0.0
    v[:40] *= 2.0 ** -990   # sums below the integer range, subnormal values among them
    flip = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]  # +j <-> -j on every axis
    a, b, c = (_call(lib.sums, x, 10) for x in (v, -v, v[:, flip]))
    assert np.array_equal(a, -b)
    odd = np.array([-1.0] * 3 + [1.0] * 4 + [-1.0] * 3)
    assert np.array_equal(a, c * odd)
    # the first sums alone are those of the point
    assert np.array_equal(a[40:, :3], a[40:, 7:])


def test_zeros_of_either_sign_add_nothing(lib):
    v = np.zeros((4, 19))
    v[0, 1], v[0, 2], v[0, 4] = 0.0, -0.0, -0.0
    v[1] = -0.0
    v[2, 1], v[2, 2] = 1e-20, -1e-20
    v[3, 2], v[3, 3], v[3, 0] = -1e-30, -0.0, -0.0
    v[:, 7] = v[:, 8] = 1.0   # y
    out = _call(lib.sums, v, 10)
    assert np.all(out[:2, [0, 2, 4, 6, 7, 9]] == 0.0)
    assert out[2, 0] == 16e-20 and out[2, 4] == 0.0
    assert out[3, 0] == 8e-30 and out[3, 4] == -16e-30
    # even sums of an odd plane: the large values cancel, the rest is at most truncated
    v = np.zeros((1, 19))
    v[0, 1], v[0, 2], v[0, 3], v[0, 4], v[0, 7] = 1.0, -1.0, 1.5, -1.5, 1e-25
    out = _call(lib.sums, v, 10)[0]
    assert out[4] == 0.0 and abs(out[3]) <= 15e-25


def test_words_keep_every_value(lib):
    r = np.random.default_rng(3)
    v = r.integers(0, 2 ** 64, 20000, dtype=np.uint64).view(np.float64)
    v = np.concatenate([v, [0.0, -0.0, 5e-324, -5e-324, 2.2250738585072009e-308, -2.2250738585072014e-308, np.inf,
                            -np.inf, 1.7e308, -1e306, 2.0 ** -951, 2.0 ** 1007, 2.0 ** 1006]])
    out = _call(lib.values, v[:, None], 1)[:, 0]
    nan = np.isnan(v)
    assert np.array_equal(np.isnan(out), nan) and np.array_equal(out[~nan], v[~nan])


def test_subnormal_and_tiny_sums_are_those_of_fp64(lib):
    r = np.random.default_rng(5)
    v = r.integers(-2 ** 40, 2 ** 40, (50, 19)).astype(float) * 5e-324
    out = _call(lib.sums, v, 10)
    for i in range(len(v)):
        for q, ex in enumerate(_exact(v[i])):   # subnormal results: every partial sum is exact
            assert Fraction(out[i, q]) == ex, (i, q)


def test_error_on_smooth_data_is_no_larger_than_in_fp64(lib):
    """Waves through zero along each axis, offsets small against the wave: the root-mean-square error of each kind
    of sum, in extended precision, against that of the FP64 sums in the order of the fallback."""
    L = np.longdouble
    r = np.random.default_rng(11)
    n = 20000
    pos = np.zeros((19, 3))
    for k in range(3):
        for j in range(3):
            pos[1 + 6 * k + 2 * j, k], pos[2 + 6 * k + 2 * j, k] = j + 1, -j - 1
    kv, ph, am = r.uniform(-0.25, 0.25, (n, 2, 3)), r.uniform(0, 2 * np.pi, (n, 2)), r.uniform(-1, 1, (n, 2))
    v = sum(am[:, None, m] * np.sin(kv[:, m] @ pos.T + ph[:, None, m]) for m in range(2))
    out = _call(lib.sums, v, 10)[:, :7]
    exact = np.zeros((n, 7), dtype=L)
    for q in range(7):
        for a in range(19):
            exact[:, q] += L(int(W[q, a])) * v[:, a].astype(L)

    def fma(a, b, c):
        return (L(a) * b.astype(L) + c.astype(L)).astype(np.float64)
    ref, s = np.empty((n, 7)), [0.0, 0.0, 0.0]
    for k in range(3):
        p, m = [v[:, 1 + 6 * k + 2 * j] for j in range(3)], [v[:, 2 + 6 * k + 2 * j] for j in range(3)]
        s = [s[j] + (p[j] + m[j]) for j in range(3)]
        ref[:, k] = fma(8.0, p[0] - m[0], -(p[1] - m[1]))
        ref[:, 4 + k] = fma(-30.0, v[:, 0], fma(16.0, p[0] + m[0], -(p[1] + m[1])))
    ref[:, 3] = fma(-60.0, v[:, 0], fma(15.0, s[0], fma(-6.0, s[1], s[2])))
    rms = lambda x: np.sqrt(np.mean((x.astype(L) - exact).astype(float) ** 2, axis=0))
    a, b = rms(out), rms(ref)
    assert np.all(a <= b), (a / b)
    # and in the worst sample
    worst = lambda x: np.abs((x.astype(L) - exact).astype(float)).max(axis=0)
    assert np.all(worst(out) <= worst(ref)), worst(out) / worst(ref)


def test_laplacian_against_exact_rationals(lib):
    for spread in (0, 4, 30, 100):
        r = np.random.default_rng(spread)
        v = r.uniform(1.0, 2.0, (200, 7)) * 2.0 ** -r.integers(0, spread + 1, (200, 7)).astype(float)
        v *= r.choice([-1.0, 1.0], v.shape)
        out, neg, e = _call(lib.laplacian, v, 1)[:, 0], _call(lib.laplacian, -v, 1)[:, 0], _exponent(v)
        assert np.array_equal(out, -neg)
        w = np.array([-6, 1, 1, 1, 1, 1, 1])
        for i in range(len(v)):
            ex = sum((int(a) * Fraction(x) for a, x in zip(w, v[i])), Fraction(0))
            top = int(e[i].max())
            bar = Fraction(2) ** (top - 56) * int(np.abs(w)[e[i] < top - 4].sum()) + abs(ex) * Fraction(1, 2 ** 53)
            assert abs(Fraction(out[i]) - ex) <= bar, i
