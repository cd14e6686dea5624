"""The fused 1D steps of the work queue in warp tasks (64 faces or cells of a field, 31 cells of the update)
give the bits of the per-stage kernels at the ends of their tasks and tiles: lines of 6 cells, one cell
around 100, 228 and 484 cells, and enough lines that each automatic tile is chosen."""
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


def _lines(ns, m, seed):
    g = np.random.default_rng(seed)
    out = []
    for n in ns:
        x = (np.arange(n) + 0.5) / n
        u = 1.0 + 0.3 * np.sin(2 * np.pi * x + g.uniform(0, 6)) + 0.4 * (x > g.uniform(0.2, 0.8))
        out.append(u[None] if m == 1 else np.stack([u, 0.2 * u, 2.0 + u]))
    return out


@pytest.mark.parametrize("m,bc", [(1, 0), (1, 1), (1, 2), (3, 0), (3, 1)])
@pytest.mark.parametrize("copies", [1, 40, 400])
def test_fused_steps_equal_the_per_stage_kernels(npw, m, bc, copies):
    ns = [6, 7, 61, 64, 99, 100, 101, 227, 229, 483, 485, 1000] * copies
    kind = npw.NPW_FLUX_EULER1D if m == 3 else npw.NPW_FLUX_BURGERS
    u0 = torch.tensor(np.concatenate([u.ravel() for u in _lines(ns, m, m + bc)]), dtype=torch.float32, device="cuda")
    p = npw.Params(rbf=npw.NPW_RBF_GA, precision=1, batch_mode=1, eta_max=1.0, inflow=(1.2, 0, 0, 0))
    specs = [dict(kind=kind, nx=n, dx=1.0 / n, t_end=0.9 / n, cfl=0.4, bc=bc) for n in ns]
    qt, _, _ = npw.make_queue_instances(specs)
    a = u0.clone()
    st, qs = npw.npweno_queue_solve(a, qt, p)
    bt, _ = npw.make_instances(ns, [1.0 / n for n in ns], [0.9 / n for n in ns], [0.4] * len(ns), [bc] * len(ns), m=m)
    b = u0.clone()
    st2, bs = npw.npweno_batch_solve(b, bt, m, kind, p)
    assert st == 0 and st2 == 0
    assert torch.equal(a, b)
    assert all(x["steps"] == y["steps"] and x["eta"] == y["eta"] for x, y in zip(qs, bs))
