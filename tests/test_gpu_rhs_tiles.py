"""ccz4_rhs leaves the halo tiles and mixed derivatives of its input in TILE and MIX, as ccz4_fill_halos_for does
(callers go on with them, ccz4_constraints_noalloc for one), on levels and meshes and in both precisions."""
import numpy as np
import pytest

from gpu_common import random_state
from paper_2406_11626_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("p,side,boxes", [(9, 2, None), (6, 3, None), (8, 2, None), (6, 4, [((1, 1, 1), (3, 3, 3))]),
                                          (9, 4, [((1, 1, 1), (3, 3, 3))])])
def test_rhs_leaves_the_tiles_of_its_input(p, side, boxes, prec):
    from paper_2406_11626_gb300 import ccz4 as C
    if boxes:
        cfg = I.multilevel_puncture_config(p=p, n_side=side, half_width=1.2, boxes=boxes)
        U, G = I.initial_state(cfg)
        U = U + np.random.default_rng(3).uniform(-1e-3, 1e-3, U.shape)
    else:
        cfg = I.single_puncture_config(p=p, n_side=side, half_width=1.0)
        U, G = random_state(p, cfg.np, cfg.origin, cfg.dx, cfg.ijk(), 3, "sommerfeld", amp=0.01, base="puncture")
    P = C.make_params(**cfg.params, precision=prec)
    g = C.Grid.from_config(cfg)
    g.upload(U, G)
    g.upload(U, G, buf="INI")
    g.fill_halos("U", P=P)
    tiles, mix = g.download("TILE"), g.download("MIX")
    for buf in ("TILE", "MIX"):
        g.as_tensor(buf).zero_()
    g.rhs(P, "U", "RHS")
    np.testing.assert_array_equal(g.download("TILE").view(np.int64), tiles.view(np.int64))
    n = g.n_points
    a, b = g.download("MIX").reshape(-1), mix.reshape(-1)
    if prec == "mixed":  # 27 FP32 slots, then alpha's and phi's in their FP64 places
        a, b = [np.concatenate([x.view(np.float32)[:27 * n].astype(float), x[18 * n:21 * n], x[30 * n:]]) for x in (a, b)]
    np.testing.assert_array_equal(a, b)
    g.close()
