"""The fixed-edge derivative pass with first derivatives outside the integer range (tiny, huge, infinite, NaN) in a
field whose mixed derivatives are taken from them: flat space with a shift of such values, whose right-hand sides are
linear in it, against the oracle. One patch of the grid only, or all of it."""
import numpy as np
import pytest

from gpu_common import both_params, make_pair
from paper_2406_11626_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,npv", [(6, (3, 2, 2)), (9, (3, 1, 2)), (9, (8, 19, 2)), (12, (2, 1, 1))])
@pytest.mark.parametrize("scale", [1e-300, 1e-309, 1e304])
@pytest.mark.parametrize("everywhere", [True, False])
def test_derivatives_of_tiny_and_huge_shifts(p, npv, scale, everywhere):
    gg, og, ijk = make_pair(p, npv, (0.0, 0.0, 0.0), 1.0, "periodic")
    U = I.flat((len(ijk), p, p, p))
    r = np.random.default_rng(p)
    for f in ("betax", "betay", "betaz"):
        q = r.uniform(-1, 1, U[0].shape)
        U[I.IDX[f]] = scale * q if everywhere else 0.0
        if not everywhere:
            U[I.IDX[f], 1] = scale * q[1]
    P, OP = both_params(**dict(I.PUNCTURE_PARAMS, ko_eps=0.3))
    gg.upload(U)
    gg.rhs(P, "U", "RHS")
    with np.errstate(all="ignore"):
        a, b = gg.download("RHS")[0], og.rhs(OP, U)[0]
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    for f in ("Ghatx", "Ghaty", "Ghatz"):
        v = I.IDX[f]
        m = np.isfinite(b[v])
        assert m.any() and np.abs(b[v][m]).max() > 0.01 * scale
        # FP64 sums of 50 terms, and the smallest numbers' own steps
        assert np.abs(a[v][m] - b[v][m]).max() <= 1e-13 * np.abs(b[v][m]).max() + 1e-321, f
    gg.close()


@pytest.mark.parametrize("p,npv", [(6, (2, 2, 1)), (9, (2, 1, 2)), (12, (1, 1, 2))])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_one_value_that_is_not_finite(p, npv, value):
    gg, og, ijk = make_pair(p, npv, (0.0, 0.0, 0.0), 0.1, "periodic")
    U = I.random_noise((len(ijk), p, p, p), seed=1, amp=1e-3)
    U[I.IDX["betay"], 0, p // 2, 0, p - 1] = value
    P, OP = both_params(**dict(I.PUNCTURE_PARAMS, ko_eps=0.3))
    gg.upload(U)
    gg.rhs(P, "U", "RHS")
    with np.errstate(all="ignore"):
        a, b = gg.download("RHS")[0], og.rhs(OP, U)[0]
    assert np.array_equal(np.isfinite(a), np.isfinite(b)) and not np.isfinite(b).all()
    m = np.isfinite(b)
    assert np.abs(a[m] - b[m]).max() <= 1e-11 * np.abs(b[m]).max()
    gg.close()
