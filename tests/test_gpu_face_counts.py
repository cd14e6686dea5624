"""Every face of a line is counted once in npw_solve_stats: switch + eval = 3 (n + 1) m per step, and in
FP64 all four counts are the oracle's, at the lengths where the last face falls beside a warp's block
(62 cells in float, 30 in double): whole lines, last slices of a cluster and last tiles of that length."""
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


def _line(n, m):
    x = (np.arange(n) + 0.5) / n
    u = 1.0 + 0.3 * np.sin(2 * np.pi * x + 0.3) + 0.2 * (x > 0.45)
    return u[None] if m == 1 else np.stack([u, 0.1 * u, 2.5 + 0.2 * u])


def _run(npw, path, u0, kind, bc, t_end, p):
    m, n = u0.shape
    u = torch.tensor(u0, dtype=torch.float32 if p.precision else torch.float64, device="cuda")
    if path == "solve":
        return npw.npweno_solve(u, 1.0 / n, t_end, 0.4, kind, bc, p)
    if path == "batch":
        table, _ = npw.make_instances([n], [1.0 / n], [t_end], [0.4], [bc], m=m)
        return npw.npweno_batch_solve(u.reshape(-1), table, m, kind, p)[1][0]
    table, _, _ = npw.make_queue_instances([dict(kind=kind, nx=n, dx=1.0 / n, t_end=t_end, cfl=0.4, bc=bc)])
    return npw.npweno_queue_solve(u.reshape(-1), table, p)[1][0]


def _total(s):
    return s["eta"]["switch"] + s["eta"]["eval"]


# float: resident (batch, queue) and cluster (solve; 16 slices, the last of 62 k, 62 k + 1 and + 2 cells)
@pytest.mark.parametrize("m", [1, 3])
@pytest.mark.parametrize("path,n", [(p, n) for p in ("batch", "queue", "solve") for n in (61, 62, 63, 64, 124, 125, 126, 187)] +
                         [("solve", n) for n in (1007, 1008, 1009, 1023, 1038, 1999, 2000)])
def test_float_lines_count_each_face_once(npw, path, n, m):
    kind, bc = (npw.NPW_FLUX_EULER1D, 1) if m == 3 else (npw.NPW_FLUX_BURGERS, 0)
    p = npw.Params(precision=1, eta_max=0.05)
    s = _run(npw, path, _line(n, m), kind, bc, 1.9 / n, p)
    assert s["steps"] >= 2 and _total(s) == 3 * (n + 1) * m * s["steps"]
    p.batch_mode = 1  # the per-stage kernels, whose phases count by another rule
    assert _run(npw, "batch", _line(n, m), kind, bc, 1.9 / n, p)["eta"] == s["eta"]


# double: the work queue (tiles of 60 cells and more), the cluster (last slices of 30, 31, 32, 61 and 91
# cells) and the per-stage kernels (a last tile of 31 and 61 cells of 1024 + .., whole lines)
@pytest.mark.parametrize("m", [1, 3])
@pytest.mark.parametrize("path,n,tile", [("queue", n, t) for n in (30, 31, 32, 61, 91, 121) for t in (0, 256)] +
                         [("solve", n, 0) for n in (31, 495, 496, 497, 511, 526, 976, 1456)] +
                         [("batch", n, t) for n in (31, 91, 1024 + 30, 1024 + 31, 1024 + 61) for t in (0, 1024)])
def test_double_counts_are_the_oracles(npw, path, n, tile, m):
    kind, bc = (npw.NPW_FLUX_EULER1D, 1) if m == 3 else (npw.NPW_FLUX_BURGERS, 0)
    u0 = _line(n, m)
    s = _run(npw, path, u0, kind, bc, 1.9 / n, npw.Params(eta_max=0.05, eta_guard=1e-3, tile_1d=tile))
    _, ref = O.solve(u0, 1.0 / n, 1.9 / n, 0.4, kind, bc, O.Params(eta_max=0.05, eta_guard=1e-3))
    assert s["steps"] == ref["steps"] >= 2 and _total(s) == 3 * (n + 1) * m * s["steps"]
    assert s["eta"] == ref["eta"]
