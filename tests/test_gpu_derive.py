"""The derivative pass and the algebra kernel that reads it, against the
oracle at the sizes where they can go wrong: patch edges around the tile
layouts (one point, the edge compiled in, the last edge whose exponents fit
in shared memory and the first whose do not), few patches (fields split over
blocks) and many, noise that uses every stencil weight, values of every
magnitude, and non-finite ones."""
import numpy as np
import pytest

import oracle as O
from gpu_common import both_params, make_pair, random_state, rel_err
from paper_2406_11626_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PUNC = dict(I.PUNCTURE_PARAMS, ko_eps=0.3)


@pytest.mark.parametrize("bc", ["periodic", "sommerfeld"])
@pytest.mark.parametrize("p,npv", [(1, (5, 4, 3)), (3, (2, 1, 3)), (8, (2, 1, 2)), (9, (1, 2, 1)), (10, (1, 1, 2)),
                                   (16, (1, 1, 1)), (17, (1, 1, 1)), (18, (1, 1, 1))])
def test_rhs_over_patch_edges(p, npv, bc):
    dx = 0.11
    origin = tuple(-0.5 * n * p * dx + 0.013 for n in npv)
    gg, og, ijk = make_pair(p, npv, origin, dx, bc)
    U = I.random_noise((len(ijk), p, p, p), seed=p, amp=1e-2)
    G = I.random_noise((gg.n_ghost,), seed=p + 1, amp=1e-2) if bc == "sommerfeld" else np.zeros((I.NV, 0))
    P, OP = both_params(**PUNC)
    gg.upload(U, G)
    gg.upload(U, G, buf="INI") if bc == "sommerfeld" else None
    gg.rhs(P, "U", "RHS")
    gU, gG = gg.download("RHS")
    rU, rG = og.rhs(OP, U, G, G)
    assert rel_err(gU, rU).max() < 1e-11 and rel_err(gG, rG).max() < 1e-11


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-13), ("mixed", 1e-7)])
def test_stages_from_filled_tiles_equal_the_step(prec, bar):
    """rk_stage takes its derivatives from the tiles of a halo fill, a step
    straight from the state: the same values."""
    from paper_2406_11626_gb300 import ccz4 as C
    cfg = I.single_puncture_config(p=9, n_side=2, half_width=1.0)
    U, G = random_state(9, cfg.np, cfg.origin, cfg.dx, cfg.ijk(), 3, "sommerfeld", amp=0.01, base="puncture")
    P = C.make_params(**cfg.params, precision=prec)
    out = []
    for stages in (False, True):
        g = C.Grid.from_config(cfg)
        g.upload(U, G)
        g.upload(U, G, buf="INI")
        if stages:
            for s in range(4):
                g.rk_stage(P, s, cfg.dt)
        else:
            g.step(P, cfg.dt, 1)
        out.append(g.download("U"))
    assert rel_err(out[0][0], out[1][0]).max() < bar and rel_err(out[0][1], out[1][1]).max() < bar


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1e305])
def test_values_beyond_the_integer_range(value):
    """One value of b^x outside the range of the integer sums, with the zero
    shift (b's right-hand side is pure dissipation): the points and values
    that the oracle has."""
    dx, p, npv = 0.1, 9, (2, 1, 1)
    gg, og, ijk = make_pair(p, npv, (0.0, 0.0, 0.0), dx, "periodic")
    U = I.random_noise((len(ijk), p, p, p), seed=1, amp=1e-2)
    U[I.IDX["bx"], 0, 4, 4, 4] = value
    P, OP = both_params(**dict(PUNC, shift="zero"))
    gg.upload(U)
    gg.rhs(P, "U", "RHS")
    a = gg.download("RHS")[0]
    with np.errstate(all="ignore"):
        b, _ = og.rhs(OP, U)
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    v = I.IDX["bx"]
    fin = np.isfinite(b[v])
    assert not fin.all() or value == 1e305
    assert np.abs(a[v][fin] - b[v][fin]).max() <= 1e-13 * np.abs(b[v][fin]).max()
    other = [q for q in range(I.NV) if q != v]
    assert rel_err(np.where(np.isfinite(b), a, 0.0), np.where(np.isfinite(b), b, 0.0))[other].max() < 1e-11


def test_fields_of_every_magnitude():
    """Dissipation of fields scaled by powers of ten from 1e-250 to 1e250."""
    dx, p, npv = 0.1, 6, (2, 2, 1)
    gg, og, ijk = make_pair(p, npv, (0.0, 0.0, 0.0), dx, "periodic")
    U = I.random_noise((len(ijk), p, p, p), seed=2, amp=1e-2)
    r = np.random.default_rng(4)
    for f, s in zip(("bx", "by", "bz"), (-250, 250, 100)):
        U[I.IDX[f]] = r.uniform(-1, 1, U[0].shape) * 10.0 ** s
    P, OP = both_params(**dict(PUNC, shift="zero"))
    gg.upload(U)
    gg.rhs(P, "U", "RHS")
    a, b = gg.download("RHS")[0], og.rhs(OP, U)[0]
    for f in ("bx", "by", "bz"):
        v = I.IDX[f]
        assert np.abs(a[v] - b[v]).max() <= 1e-13 * np.abs(b[v]).max(), f
