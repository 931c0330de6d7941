"""FP64 stages with the derivative pass beside the algebra in one launch, against
the two launches of the same grid: the same bits, from the smallest grid that
takes the one launch over a last round of few patches to refined meshes; and
the derivative pass of the other fixed patch edges against the oracle."""
import numpy as np
import pytest

from gpu_common import both_params, make_pair, rel_err
from paper_2406_11626_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PUNC = dict(I.PUNCTURE_PARAMS, ko_eps=0.3)


def _noise(grid, seed):
    """Noise around flat space, the last field's from 1e-300 to 1 (values below and within the integer range)."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = grid.as_tensor("U").view(I.NV, grid.field_stride)
    u.copy_(1e-2 * (2.0 * torch.rand(u.shape, generator=gen, device="cuda", dtype=torch.float64) - 1.0))
    for v in (0, 3, 5, 6, 10):  # diagonal of the metric, lapse, conformal factor
        u[v] += 1.0
    e = torch.randint(-300, 1, (grid.field_stride // 64 + 1,), generator=gen, device="cuda")
    u[24] *= torch.pow(10.0, e.double()).repeat_interleave(64)[:grid.field_stride]
    if grid.n_ghost:
        grid.as_tensor("INI").copy_(grid.as_tensor("U"))
    return grid.as_tensor("U").clone()


def _same(grid, P, dt, seed):
    import torch
    start, out = _noise(grid, seed), []
    # one launch, two launches, two launches with the work counter
    for shape, mode in ((0, "flat"), (3, "flat"), (0, "queue")):
        grid.set_tuning(shape, 0)
        grid.set_launch(mode)
        grid.as_tensor("U").copy_(start)
        grid.step(P, dt, 1)
        grid.step_graph(P, dt, 1)
        torch.cuda.synchronize()
        u = grid.as_tensor("U").view(I.NV, grid.field_stride)
        out.append(u[:, :grid.n_points + grid.n_ghost].clone())
    assert bool(torch.isfinite(out[0]).all())
    for other in out[1:]:
        assert torch.equal(out[0].view(torch.int64), other.view(torch.int64))


@pytest.mark.parametrize("npv,bc", [((8, 19, 2), "periodic"), ((8, 19, 2), "sommerfeld"), ((7, 7, 11), "sommerfeld"),
                                    ((10, 9, 9), "periodic"), ((5, 5, 43), "sommerfeld")])
def test_one_launch_equals_two(npv, bc):
    from paper_2406_11626_gb300 import ccz4 as C
    grid = C.Grid(9, npv, I.patch_ijk(npv), tuple(-0.5 * 9 * n * 0.11 + 0.013 for n in npv), 0.11, bc)
    _same(grid, C.make_params(**PUNC), 0.01, 7)
    grid.close()


def test_one_launch_equals_two_on_a_mesh():
    from paper_2406_11626_gb300 import ccz4 as C
    level, ijk = I.refined_mesh((7,) * 3, [((1,) * 3, (5, 4, 5))])  # 1639 patches: meshes below about 1100 keep two launches
    cfg = I.MeshConfig(name="", p=9, np=(7,) * 3, origin=(-3.4,) * 3, dx=0.11, bc="sommerfeld", params=PUNC, dt=0.003,
                       steps=1, level=level, mesh_ijk=ijk)
    grid = C.Grid.from_config(cfg)
    _same(grid, C.make_params(**PUNC), cfg.dt, 8)
    grid.close()


@pytest.mark.parametrize("p,npv", [(6, (1, 1, 1)), (6, (3, 2, 4)), (12, (1, 1, 1)), (12, (2, 1, 2))])
@pytest.mark.parametrize("bc", ["periodic", "sommerfeld"])
def test_rhs_of_fixed_patch_edges(p, npv, bc):
    dx = 0.11
    gg, og, ijk = make_pair(p, npv, tuple(-0.5 * n * p * dx + 0.013 for n in npv), dx, bc)
    U = I.random_noise((len(ijk), p, p, p), seed=p, amp=1e-2)
    G = I.random_noise((gg.n_ghost,), seed=p + 1, amp=1e-2) if bc == "sommerfeld" else np.zeros((I.NV, 0))
    P, OP = both_params(**PUNC)
    gg.upload(U, G)
    gg.upload(U, G, buf="INI") if bc == "sommerfeld" else None
    gg.rhs(P, "U", "RHS")
    gU, gG = gg.download("RHS")
    rU, rG = og.rhs(OP, U, G, G)
    assert rel_err(gU, rU).max() < 1e-11 and rel_err(gG, rG).max() < 1e-11
