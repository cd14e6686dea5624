"""Characteristic runs on a state whose Roe average at some faces has no real sound speed: those faces take no
shape-parameter decision.  Their flag bytes are 0, and with switch, guard and bound off no such decision is
counted while the run ends as not finite."""
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


def _state(n):
    g = np.random.default_rng(n)
    rho, v = 1.0 + 0.1 * g.uniform(size=n), 0.3 * g.normal(size=n)
    E = 2.5 + 0.5 * rho * v * v
    E[n // 3: n // 2] = -1.0  # negative pressure
    return np.stack([rho, rho * v, E])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("k", [2, 3])
@pytest.mark.parametrize("n", [60, 3000])
def test_faces_without_a_roe_state_take_no_decision(npw, precision, k, n):
    u0 = torch.tensor(_state(n), dtype=torch.float32 if precision else torch.float64, device="cuda")
    p = npw.Params(precision=precision, k=k, characteristic=1, monotone_switch=0, eta_guard=-1.0, tie_tol=0.1)
    vm, vp, fl, eta = npw.npweno_reconstruct(u0, 1, p, True, True)
    bad = torch.isnan(vm)
    assert bad.any() and not bad.all() and torch.equal(bad, torch.isnan(vp)) and torch.isnan(eta[bad]).all()
    assert not fl[bad].any() and not (fl & 0xC9).any()
    u = u0.clone()
    table, _ = npw.make_instances([n], [1.0 / n], [1.0], [0.4], [1], m=3)
    st, s = npw.npweno_batch_solve(u.reshape(-1), table, 3, npw.NPW_FLUX_EULER1D, p, raise_on_error=False)
    assert st == npw.NPW_ENONFINITE and s[0]["steps"] >= 0
    c = s[0]["eta"]
    assert (c["switch"], c["guard"], c["bound"]) == (0, 0, 0)
    assert c["eval"] == 3 * (3 if k == 3 else 6) * (n + 1) * s[0]["steps"]
