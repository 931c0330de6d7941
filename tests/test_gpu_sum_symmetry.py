"""The stencil sums on the GPU keep the symmetries that FP64 sums have: with the
zero shift the right-hand side of b is pure dissipation, a sum over the 19 points
of a field alone, so its sign follows the field's bit for bit, at every magnitude
and beside zeros of either sign, for each body of the derivative pass (the fixed
edges 6, 9 and 12, one field or several to a block, the general one)."""
import numpy as np
import pytest

from paper_2406_11626_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,npv", [(6, (2, 2, 2)), (9, (3, 1, 2)), (9, (5, 8, 8)), (8, (2, 2, 1)), (12, (2, 1, 2)),
                                   (18, (1, 1, 1))])
def test_dissipation_is_odd(p, npv):
    from paper_2406_11626_gb300 import ccz4 as C
    ijk = I.patch_ijk(npv)
    P = C.make_params(**dict(I.PUNCTURE_PARAMS, shift="zero", ko_eps=0.3))
    U = I.random_noise((len(ijk), p, p, p), seed=p, amp=1e-2)
    r = np.random.default_rng(p)
    for f in ("bx", "by", "bz"):
        q = r.uniform(-1, 1, U[0].shape) * 10.0 ** -r.integers(0, {"bx": 2, "by": 25, "bz": 200}[f], U[0].shape)
        q[r.random(q.shape) < 0.05] = 0.0
        q[r.random(q.shape) < 0.05] = -0.0
        U[I.IDX[f]] = q
    out = []
    for s in (1.0, -1.0):
        V = U.copy()
        V[I.IDX["bx"]:I.IDX["bz"] + 1] *= s
        g = C.Grid(p, npv, ijk, (0.0, 0.0, 0.0), 0.1, "periodic")
        g.upload(V)
        g.rhs(P, "U", "RHS")
        out.append(g.download("RHS")[0][I.IDX["bx"]:I.IDX["bz"] + 1])
        g.close()
    assert np.all(np.isfinite(out[0])) and np.abs(out[0]).max() > 0
    assert np.array_equal(out[0], -out[1])
