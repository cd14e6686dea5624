"""The automatic tile of the 1D per-stage kernels (32 w - halo cells, chosen from the number of
cells so that short lines spread over the SMs) gives the bits of an explicit 1024-cell tile, at the
edges of the rule: lines shorter than one tile, one cell around a tile's end, and several waves of
tiles; a batch's tile table holds the smaller tiles."""
import numpy as np
import pytest

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


def _line(n, m, seed):
    g = np.random.default_rng(seed)
    x = (np.arange(n) + 0.5) / n
    u = 1.0 + 0.3 * np.sin(2 * np.pi * x + g.uniform(0, 6)) + 0.2 * (x > 0.55)
    return u[None] if m == 1 else np.stack([u, 0.1 * u, 2.5 + 0.2 * u])


@pytest.mark.parametrize("n", [6, 29, 31, 32, 62, 63, 152 * 31, 152 * 31 + 1, 20011])
@pytest.mark.parametrize("precision,m,char", [(0, 1, 0), (0, 3, 0), (0, 3, 1), (1, 1, 0), (1, 3, 0), (1, 3, 1)])
def test_automatic_tile_gives_the_same_bits(npw, n, precision, m, char):
    dt = torch.float32 if precision else torch.float64
    kind, bc = (npw.NPW_FLUX_EULER1D, 1) if m == 3 else (npw.NPW_FLUX_BURGERS, 0)
    u0 = torch.tensor(_line(n, m, n), dtype=dt, device="cuda")
    out = []
    for tile in (0, 1024):
        u = u0.clone()
        a = npw.npweno_rk3_step(u, 1.0 / n, 0.1 / n, kind, bc, npw.Params(precision=precision, characteristic=char,
                                                                         tile_1d=tile, eta_max=1.0), want_alpha=True)
        npw.npweno_solve(u, 1.0 / n, 0.9 / n, 0.3, kind, bc, npw.Params(precision=precision, characteristic=char,
                                                                        tile_1d=tile, eta_max=1.0))
        out.append((a, u))
    assert out[0][0] == out[1][0] and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_table_holds_the_automatic_tiles(npw, precision):
    ns = [6, 40, 300, 31, 9000]
    dt = torch.float32 if precision else torch.float64
    u0 = torch.tensor(np.concatenate([_line(n, 1, n)[0] for n in ns]), dtype=dt, device="cuda")
    table, _ = npw.make_instances(ns, [1.0 / n for n in ns], [0.02] * 5, [0.5] * 5, [0] * 5)
    out = []
    for tile in (0, 256):
        u = u0.clone()
        st, _ = npw.npweno_batch_solve(u, table, 1, npw.NPW_FLUX_BURGERS,
                                       npw.Params(precision=precision, batch_mode=1, tile_1d=tile))
        assert st == 0
        out.append(u)
    assert torch.equal(out[0], out[1])
