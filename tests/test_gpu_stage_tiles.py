"""The automatic tile of the 1D per-stage kernels, reached through batch_mode 1 (short single lines take a cluster and
no tile): the bits and decision counts of an explicit 1024-cell tile, for every body -- component-wise and
characteristic, both precisions and orders -- at line lengths around the ends of its tiles (32 w - 3, 32 w - 1
and 30 w cells), alone, with the other lengths in one batch, and beside resident instances."""
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


def _batch(npw, ns, m, p):
    kind, bc = (npw.NPW_FLUX_EULER1D, 1) if m == 3 else (npw.NPW_FLUX_BURGERS, 0)
    dt = torch.float32 if p.precision else torch.float64
    u = torch.tensor(np.concatenate([_line(n, m, n).ravel() for n in ns]), dtype=dt, device="cuda")
    table, _ = npw.make_instances(ns, [1.0 / n for n in ns], [0.9 / n for n in ns], [0.3] * len(ns), [bc] * len(ns), m=m)
    st, stats = npw.npweno_batch_solve(u, table, m, kind, p)
    assert st == 0
    return u, stats


BODIES = [(k, precision, m, char) for k in (2, 3) for precision in (0, 1) for m, char in ((1, 0), (3, 0), (3, 1))]


@pytest.mark.parametrize("k,precision,m,char", BODIES)
@pytest.mark.parametrize("n", [6, 29, 30, 31, 32, 61, 62, 63, 125, 126, 152 * 31, 152 * 31 + 1, 20011, 152 * 509 + 1])
def test_lines_of_one_length(npw, n, k, precision, m, char):
    out = [_batch(npw, [n], m, npw.Params(k=k, precision=precision, characteristic=char, batch_mode=1, tile_1d=tile,
                                          eta_max=1.0)) for tile in (0, 1024)]
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


@pytest.mark.parametrize("k,precision,m,char", BODIES)
@pytest.mark.parametrize("mode", [0, 1])
def test_lines_together(npw, k, precision, m, char, mode):
    ns = [6, 31, 63, 254, 255, 509, 510, 1021, 1022, 20011] + [70] * 160
    out = [_batch(npw, ns, m, npw.Params(k=k, precision=precision, characteristic=char, batch_mode=mode, tile_1d=tile,
                                         eta_max=1.0)) for tile in (0, 256, 1024)]
    for u, stats in out[1:]:
        assert torch.equal(u, out[0][0]) and stats == out[0][1]


@pytest.mark.parametrize("m", [1, 3])
@pytest.mark.parametrize("ns", [[40], [129], [3000, 500], [20000, 9000, 257], [152 * 512 + 1], [152 * 1024]])
def test_fused_steps_of_k2(npw, ns, m):
    """The automatic tile of the queue's fused k = 2 steps (64 to 1024 cells) against 256 cells."""
    kind, bc = (npw.NPW_FLUX_EULER1D, 1) if m == 3 else (npw.NPW_FLUX_BURGERS, 0)
    specs = [dict(kind=kind, nx=n, dx=1.0 / n, t_end=0.9 / n, cfl=0.3, bc=bc) for n in ns]
    table, _, _ = npw.make_queue_instances(specs)
    u0 = torch.tensor(np.concatenate([_line(n, m, n).ravel() for n in ns]), dtype=torch.float32, device="cuda")
    out = []
    for tile in (0, 256):
        u = u0.clone()
        st, stats = npw.npweno_queue_solve(u, table, npw.Params(k=2, precision=1, batch_mode=1, tile_1d=tile, eta_max=1.0))
        assert st == 0
        out.append((u, stats))
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
