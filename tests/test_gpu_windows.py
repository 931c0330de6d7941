"""Grids whose derivative buffer holds a part of their patches (CCZ4_DERIVE_POINTS, or memory too short for more):
every call that takes derivatives gives the bits that it gives with a buffer for all patches."""
import numpy as np
import pytest

from paper_2406_11626_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PUNC = dict(I.PUNCTURE_PARAMS, ko_eps=0.3)


def _fill(grid, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = grid.as_tensor("U").view(I.NV, grid.field_stride)
    u.copy_(1e-2 * (2.0 * torch.rand(u.shape, generator=gen, device="cuda", dtype=torch.float64) - 1.0))
    for v in (0, 3, 5, 6, 10):  # diagonal of the metric, lapse, conformal factor
        u[v] += 1.0
    if grid.n_ghost:
        grid.as_tensor("INI").copy_(grid.as_tensor("U"))


def _calls(grid, mixed):
    """Everything that reads the derivative buffer, on the same state."""
    import torch
    from paper_2406_11626_gb300 import ccz4 as C
    P = C.make_params(**PUNC, precision="mixed" if mixed else "fp64")
    out, n = [], grid.n_points + grid.n_ghost

    def keep(buf):
        torch.cuda.synchronize()
        out.append(grid.as_tensor(buf).view(I.NV, grid.field_stride)[:, :n].clone())
    for mode in ("flat", "queue") + (("fused",) if grid.p == 9 else ()):
        grid.set_launch(mode)
        _fill(grid, 5)
        grid.step(P, 0.003, 1)
        grid.step_graph(P, 0.003, 1)
        keep("U")
    grid.set_launch("flat")
    for shape in (1, 3):
        grid.set_tuning(shape, 0)
        _fill(grid, 5)
        grid.step(P, 0.003, 1)
        keep("U")
    grid.set_tuning(0, 0)
    _fill(grid, 5)
    grid.rhs(P, "U", "RHS")
    keep("RHS")
    for s in range(4):
        grid.rk_stage(P, s, 0.003)
    keep("U")
    if not mixed:
        H = torch.empty(grid.n_points, dtype=torch.float64, device="cuda")
        M = torch.empty(3 * grid.n_points, dtype=torch.float64, device="cuda")
        out.append(torch.as_tensor(grid.constraints("U", H.data_ptr(), M.data_ptr())))
        out += [H, M, grid.as_tensor("TILE").clone(), grid.as_tensor("MIX").clone()]
        grid.psi4("U", "RHS", (0.01, 0.02, 0.03))
        torch.cuda.synchronize()
        out.append(grid.as_tensor("RHS").view(I.NV, grid.field_stride)[:2, :grid.n_points].clone())
    return out


def _same(a, b):
    import torch
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert bool(torch.isfinite(x).all()) and torch.equal(x.view(torch.int64), y.view(torch.int64))


# (patch edge, patches per axis, patches that the buffer may hold)
LEVELS = [(9, (8, 19, 4), 400), (9, (8, 19, 4), 200), (9, (5, 8, 8), 256), (6, (5, 4, 4), 32), (12, (3, 2, 2), 4),
          (8, (2, 2, 3), 1), (5, (7, 6, 7), 256)]


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("p,npv,hold", LEVELS)
def test_windows_of_a_level(p, npv, hold, mixed, monkeypatch):
    from paper_2406_11626_gb300 import ccz4 as C
    out = []
    for points in ("", str(hold * p ** 3)):
        monkeypatch.setenv("CCZ4_DERIVE_POINTS", points)
        g = C.Grid(p, npv, I.patch_ijk(npv), tuple(-0.5 * n * p * 0.11 + 0.013 for n in npv), 0.11, "sommerfeld")
        out.append(_calls(g, mixed))
        g.close()
    _same(*out)


@pytest.mark.parametrize("mixed", [False, True])
def test_windows_of_a_mesh(mixed, monkeypatch):
    from paper_2406_11626_gb300 import ccz4 as C
    level, ijk = I.refined_mesh((6,) * 3, [((2,) * 3, (5, 4, 5))])
    out = []
    for points in ("", str(256 * 729)):
        monkeypatch.setenv("CCZ4_DERIVE_POINTS", points)
        g = C.Grid(9, (6,) * 3, ijk, (-2.9,) * 3, 0.11, "sommerfeld", level=level)
        out.append(_calls(g, mixed))
        g.close()
    _same(*out)


@pytest.mark.parametrize("variant", ["fo", "so-recon"])
@pytest.mark.parametrize("p,npv,hold", [(9, (7, 6, 7), 256), (6, (4, 4, 4), 32)])
def test_windows_of_the_58_variable_formulations(p, npv, hold, variant, monkeypatch):
    from paper_2406_11626_gb300 import ccz4 as C
    r = np.random.default_rng(2)
    n = npv[0] * npv[1] * npv[2]
    U = 1e-3 * r.uniform(-1, 1, (I.NV_FO, n, p, p, p))
    for v in (0, 3, 5, 6, 10):
        U[v] += 1.0
    P = C.make_params(**PUNC)
    out = []
    for points in ("", str(hold * p ** 3)):
        monkeypatch.setenv("CCZ4_DERIVE_POINTS", points)
        g = C.Grid(p, npv, I.patch_ijk(npv), tuple(-0.5 * k * p * 0.11 + 0.013 for k in npv), 0.11, "sommerfeld")
        f = C.FirstOrder(g, variant)
        G = np.zeros((I.NV_FO, g.n_ghost))
        G[[0, 3, 5, 6, 10]] = 1.0
        f.upload(U, G)
        f.upload(U, G, buf="INI")
        f.step(P, 0.003, 1)
        f.rhs(P, "U", "RHS")
        out.append(f.download("U") + f.download("RHS"))
        f.close()
        g.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)


def test_a_grid_is_made_where_memory_is_short():
    """An allocator that refuses the derivative buffer of all patches: the grid takes a smaller one and steps alike;
    one that refuses the other buffers' sizes too: the error, as ever."""
    import torch
    from paper_2406_11626_gb300 import ccz4 as C
    p, npv = 9, (10, 8, 8)
    points = npv[0] * npv[1] * npv[2] * p ** 3
    limit, asked = [1 << 62], []

    def alloc(ctx, nbytes, stream):
        asked.append(nbytes)
        return torch.cuda.caching_allocator_alloc(int(nbytes)) if nbytes <= limit[0] else None

    def dealloc(ctx, ptr, nbytes, stream):
        torch.cuda.caching_allocator_delete(int(ptr))
    cbs = (C._ALLOC_FN(alloc), C._DEALLOC_FN(dealloc))
    P, out = C.make_params(**PUNC), []
    assert C.lib().ccz4_set_allocator(cbs[0], cbs[1], None) == C.OK
    try:
        for per_point in (1000, 120):  # doubles: the derivatives take 133 a point, the tiles 116
            limit[0], asked[:] = 8 * per_point * points, []
            g = C.Grid(p, npv, I.patch_ijk(npv), (0.0, 0.0, 0.0), 0.1, "periodic")
            assert (max(asked) > limit[0]) == (per_point == 120)
            _fill(g, 1)
            g.step(P, 0.003, 1)
            torch.cuda.synchronize()
            out.append(g.as_tensor("U").clone())
            g.close()
        limit[0] = 8 * 20 * points
        with pytest.raises(C.CCZ4Error) as e:
            C.Grid(p, npv, I.patch_ijk(npv), (0.0, 0.0, 0.0), 0.1, "periodic")
        assert e.value.code == C.ERR_NOMEM
    finally:
        C.lib().ccz4_set_allocator(C._ALLOC_FN(), C._DEALLOC_FN(), None)
    assert torch.equal(out[0].view(torch.int64), out[1].view(torch.int64))
