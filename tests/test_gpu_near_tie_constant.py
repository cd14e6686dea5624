"""Near-tie flags of constant stencils.  In NPW_FP64 the numerator and the denominator of a constant stencil
are the round-off of 3 w and 15 w, so that eta and the denominator may lie at the bound or at a guard of
round-off size; on float data both are exactly 0 and no threshold is near."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("eps_M,bound,guard,tol", [(1e-12, 1.0, 0.0, 1e-5), (0.0, 1.0, 0.0, 0.0), (1e-12, 0.0, 2.0 ** -55, 1e-5),
                                                   (1e-12, 0.0, 0.0, 1e-5), (1e-3, 0.5, 1e-3, 1e-5)])
def test_constant_stencils(npw, precision, eps_M, bound, guard, tol):
    g = np.random.default_rng(4)
    u = np.repeat(g.normal(size=500) * 10.0 ** g.uniform(-3, 8, 500), 9)
    u[900:1800] = 0.0
    if precision:
        u = u.astype(np.float32).astype(np.float64)
    n = u.size
    w0, w1, w2, w3 = (u[(np.arange(n + 1) + k) % n] for k in (-2, -1, 0, 1))
    const = (w0 == w1) & (w1 == w2) & (w2 == w3)
    p = npw.Params(precision=precision, eps_M=eps_M, eta_max=bound, eta_guard=guard or -1.0, tie_tol=tol)
    d = torch.tensor(u, dtype=torch.float32 if precision else torch.float64, device="cuda")
    fl = npw.npweno_reconstruct(d, 0, p)[2].cpu().numpy()
    t = tol or 1e-10
    rel = lambda a, b: (np.fmax(np.abs(a), np.abs(b)) > 0.0) & (np.abs(a - b) <= t * np.fmax(np.abs(a), np.abs(b)))
    near = np.zeros(n + 1, bool)
    with np.errstate(all="ignore"):
        den = w0 - 15.0 * w1 + 15.0 * w2 - w3
        if guard:
            near |= rel(np.abs(den), guard * (np.abs(w0) + 15.0 * np.abs(w1) + 15.0 * np.abs(w2) + np.abs(w3)))
        if bound:
            near |= rel(np.abs((w0 - 3.0 * w1 + 3.0 * w2 - w3) / (den + eps_M)), bound)
    assert np.array_equal(((fl & 2) != 0)[const], near[const])
    if precision == 0 and eps_M == 0.0:
        assert near[const].any()
