"""Which launches a step takes (Grid.stage_launches): the grids whose one-launch stages other tests compare with two
launches do take one, every other setting two for each window; and the shapes of a mixed step give the same bits."""
import numpy as np
import pytest

from paper_2406_11626_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PUNC = dict(I.PUNCTURE_PARAMS, ko_eps=0.3)


def _level(p, npv, bc="periodic"):
    from paper_2406_11626_gb300 import ccz4 as C
    return C.Grid(p, npv, I.patch_ijk(npv), tuple(-0.5 * p * n * 0.11 + 0.013 for n in npv), 0.11, bc)


def _params(**kw):
    from paper_2406_11626_gb300 import ccz4 as C
    return C.make_params(**PUNC, **kw)


@pytest.mark.parametrize("npv", [(8, 19, 2), (7, 7, 11), (10, 9, 9), (5, 5, 43)])
def test_large_fp64_levels_take_one_launch(npv):
    g = _level(9, npv)
    assert g.stage_launches(_params()) == 1
    assert g.stage_launches(_params(precision="mixed")) == 2
    for shape in (1, 2, 3):
        g.set_tuning(shape, 0)
        assert g.stage_launches(_params()) == 2
    g.set_tuning(0, 0)
    for mode, n in (("queue", 2), ("fused", 1), ("flat", 1)):
        g.set_launch(mode)
        assert g.stage_launches(_params()) == n
    g.close()


def test_large_fp64_meshes_take_one_launch():
    from paper_2406_11626_gb300 import ccz4 as C
    level, ijk = I.refined_mesh((7,) * 3, [((1,) * 3, (5, 4, 5))])
    g = C.Grid(9, (7,) * 3, ijk, (-3.4,) * 3, 0.11, "sommerfeld", level=level)
    assert g.stage_launches(_params()) == 1 and g.stage_launches(_params(precision="mixed")) == 2
    g.close()


@pytest.mark.parametrize("side,box,launches", [(5, (2, 2, 2), 2), (6, (2, 2, 2), 1), (8, (3, 3, 3), 1)])
def test_the_line_between_the_launches_of_meshes(side, box, launches):
    from paper_2406_11626_gb300 import ccz4 as C
    lo = [(side - b) // 2 for b in box]
    level, ijk = I.refined_mesh((side,) * 3, [(tuple(lo), tuple(a + b for a, b in zip(lo, box)))])
    g = C.Grid(9, (side,) * 3, ijk, (-3.0,) * 3, 0.11, "periodic", level=level)
    assert g.stage_launches(_params()) == launches
    g.close()


@pytest.mark.parametrize("npv,launches", [((6, 6, 7), 2), ((7, 7, 6), 1), ((7, 7, 7), 2), ((6, 8, 8), 1)])
def test_the_line_between_the_launches_of_levels(npv, launches):
    g = _level(9, npv)
    assert g.stage_launches(_params()) == launches
    g.close()


@pytest.mark.parametrize("p,npv", [(9, (3, 3, 3)), (8, (8, 8, 8)), (12, (4, 4, 4)), (6, (8, 8, 8))])
def test_other_grids_take_two(p, npv):
    g = _level(p, npv)
    assert g.stage_launches(_params()) == 2
    g.close()


def test_windows_are_counted(monkeypatch):
    monkeypatch.setenv("CCZ4_DERIVE_POINTS", str(256 * 729))
    g = _level(9, (8, 9, 8))
    assert g.stage_launches(_params()) == 6 and g.stage_launches(_params(precision="mixed")) == 6
    g.close()


def test_null_arguments_are_refused():
    from paper_2406_11626_gb300 import ccz4 as C
    g = _level(9, (2, 1, 1))
    assert C.lib().ccz4_stage_launches(g._h, None, None) == C.ERR_INVALID
    assert C.lib().ccz4_stage_launches(None, None, None) == C.ERR_INVALID
    g.close()


@pytest.mark.parametrize("p,npv", [(9, (8, 8, 5)), (7, (3, 2, 2))])
def test_shapes_of_a_mixed_step_give_the_same_bits(p, npv):
    import torch
    P, out = _params(precision="mixed"), []
    g = _level(p, npv, "sommerfeld")
    U = I.random_noise((len(g.ijk), p, p, p), seed=4, amp=1e-2)
    G = I.random_noise((g.n_ghost,), seed=5, amp=1e-2)
    for stage in (0, 1, 2, 3):
        for fill in (0, 1, 2, 3):
            g.set_tuning(stage, fill)
            g.upload(U, G)
            g.upload(U, G, buf="INI")
            g.step(P, 0.003, 1)
            torch.cuda.synchronize()
            out.append(g.download("U"))
    for o in out[1:]:
        np.testing.assert_array_equal(o[0], out[0][0])
        np.testing.assert_array_equal(o[1], out[0][1])
    g.close()
