"""The 2D warp-task body (NPW_FP32_MIXED, k = 3) at the edges of its 30 x 11 tiles: grids smaller than a
tile and one cell around a tile's end in either direction, all three flux kinds.
  * Boundaries: one RK3 step of WENO-JS from float data against the FP64 oracle, every boundary
    condition: no shape parameter, so nothing is decided from float stage values, and the result is
    within float rounding of the candidates, weights, flux and update, 2e-6 of the largest value as
    for the other mixed steps.
  * Tiles: rolling a periodic grid rolls the result, bit for bit (each cell's arithmetic depends on its
    neighbours and the wave speed only), with the shape parameter, the switch and the bound on.
  * The work queue and the single-grid entry point run the same body and give the same bits."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def npw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1602_00182_gb300 import build as b
    b.build()
    import paper_1602_00182_gb300.npweno as m
    m.load()
    return m


def _grid(kind, nx, ny):
    x, y = (np.arange(nx) + 0.3) / max(nx, 12), (np.arange(ny) + 0.6) / max(ny, 12)
    s = 1.0 + 0.3 * np.sin(2 * np.pi * x)[None, :] * np.cos(2 * np.pi * y)[:, None] + 0.1 * x[None, :]
    u = s[None] if kind != O.EULER2D else np.stack([s, 0.3 * s, -0.2 * s * s, 2.0 + s])
    return u.astype(np.float32).astype(np.float64)


SHAPES = [(6, 6), (29, 11), (30, 12), (31, 10), (32, 23), (61, 22)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("kind", [O.ADVECTION, O.BURGERS, O.EULER2D])
@pytest.mark.parametrize("bc,bc_y", [(0, 0), (1, 0), (2, 1), (0, 2)])
def test_boundaries_at_tile_edges(npw, nx, ny, kind, bc, bc_y):
    U = _grid(kind, nx, ny)
    inflow = (1.1, 0.2, 0.1, 3.0)
    d, dt = 0.05, 0.003
    op = O.Params(scheme=O.WENO_JS, inflow=inflow, bc_y=bc_y)
    ref = O.rk3_step_2d(U, d, d, dt, kind, bc, op)
    p = npw.Params(scheme=npw.NPW_WENO_JS, inflow=inflow, bc_y=bc_y, precision=1)
    g = torch.tensor(U, dtype=torch.float32, device="cuda")
    npw.npweno_rk3_step_2d(g, d, d, dt, kind, bc, p)
    e = np.abs(g.cpu().numpy().astype(np.float64) - ref)
    assert e.max() <= 2e-6 * np.abs(ref).max(), e.max()


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("kind", [O.ADVECTION, O.BURGERS, O.EULER2D])
def test_rolled_grid_gives_the_rolled_bits(npw, nx, ny, kind):
    p = npw.Params(eta_max=1.0, precision=1)
    g = torch.tensor(_grid(kind, nx, ny), dtype=torch.float32, device="cuda")
    r = torch.roll(g, (7, 5), (-1, -2)).contiguous()
    for u in (g, r):
        npw.npweno_rk3_step_2d(u, 0.05, 0.05, 0.003, kind, 0, p)
    assert torch.equal(torch.roll(g, (7, 5), (-1, -2)), r)


def test_queue_of_ragged_grids_equals_single_solves(npw):
    p = npw.Params(rbf=npw.NPW_RBF_GA, precision=1, eta_max=1.0)
    shapes = [(6, 6), (31, 12), (60, 22), (95, 37)]
    grids = [torch.tensor(_grid(O.EULER2D, nx, ny), dtype=torch.float32, device="cuda") for nx, ny in shapes]
    specs = [dict(kind=O.EULER2D, nx=nx, ny=ny, dx=0.05, dy=0.05, t_end=0.02, cfl=0.5, bc=0) for nx, ny in shapes]
    table, total, offs = npw.make_queue_instances(specs)
    arena = torch.cat([g.reshape(-1) for g in grids])
    st, stats = npw.npweno_queue_solve(arena, table, p)
    assert st == 0
    for g, off, s in zip(grids, offs, stats):
        one = npw.npweno_solve_2d(g, 0.05, 0.05, 0.02, 0.5, O.EULER2D, 0, p)
        assert torch.equal(arena[off:off + g.numel()], g.reshape(-1))
        assert one["steps"] == s["steps"] and one["eta"] == s["eta"]
