"""One line solved whole by one thread-block cluster (npweno_solve, npweno_rk3_step on short lines) gives
the bits, step counts and decision counts of the per-stage kernels: lines of one slice and of 2 to 16,
last slices of three cells and more, the ends of the warps' blocks (62 cells float, 30 double), every
boundary condition and scheme, the step limit and a state that is not finite."""
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


def _line(n, m, precision):
    x = (np.arange(n) + 0.5) / n
    u = 1.0 + 0.3 * np.sin(2 * np.pi * x + 0.3) + 0.3 * (x > 0.45)
    u = u[None] if m == 1 else np.stack([u, 0.3 * u, 2.0 + u])
    return torch.tensor(u, dtype=torch.float32 if precision else torch.float64, device="cuda")


def _per_stage(npw, u0, kind, bc, dx, t_end, cfl, p):
    u = u0.clone()
    m, n = u.shape
    table, _ = npw.make_instances([n], [dx], [t_end], [cfl], [bc], m=m)
    p.batch_mode = 1
    st, stats = npw.npweno_batch_solve(u.reshape(-1), table, m, kind, p, raise_on_error=False)
    return u, st, stats[0]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [6, 7, 8, 15, 16, 17, 31, 129, 131, 200, 480, 497, 993, 1499])
@pytest.mark.parametrize("m,bc", [(1, 0), (1, 2), (3, 1), (3, 0)])
def test_solve_equals_the_per_stage_kernels(npw, precision, n, m, bc):
    kind = npw.NPW_FLUX_EULER1D if m == 3 else npw.NPW_FLUX_BURGERS
    u0 = _line(n, m, precision)
    p = npw.Params(rbf=npw.NPW_RBF_GA, precision=precision, inflow=(1.1, 0, 0, 0), eta_max=1.0)
    ref, st, s = _per_stage(npw, u0, kind, bc, 1.0 / n, 2.3 / n, 0.4, p)
    u = u0.clone()
    got = npw.npweno_solve(u, 1.0 / n, 2.3 / n, 0.4, kind, bc, p)
    assert torch.equal(u, ref) and got == s
    # one step of a given dt: the run that ends after it
    dt = 0.1 / n
    ref, _, s = _per_stage(npw, u0, kind, bc, 1.0 / n, dt, 100.0, p)
    u = u0.clone()
    a = npw.npweno_rk3_step(u, 1.0 / n, dt, kind, bc, p, want_alpha=True)
    assert s["steps"] == 1 and torch.equal(u, ref) and a > 0.0


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("scheme", [0, 1, 2, 3])
@pytest.mark.parametrize("kind", [0, 1])
def test_schemes(npw, precision, scheme, kind):
    n = 333
    u0 = _line(n, 1, precision)
    p = npw.Params(scheme=scheme, precision=precision)
    ref, _, s = _per_stage(npw, u0, kind, 0, 1.0 / n, 0.05, 0.5, p)
    u = u0.clone()
    assert npw.npweno_solve(u, 1.0 / n, 0.05, 0.5, kind, 0, p) == s
    assert torch.equal(u, ref)


@pytest.mark.parametrize("n", [5613, 39999])
def test_long_float_lines(npw, n):
    u0 = _line(n, 1, 1)
    p = npw.Params(rbf=npw.NPW_RBF_GA, precision=1)
    ref, _, s = _per_stage(npw, u0, npw.NPW_FLUX_BURGERS, 0, 1.0 / n, 9.0 / n, 0.5, p)
    u = u0.clone()
    assert npw.npweno_solve(u, 1.0 / n, 9.0 / n, 0.5, npw.NPW_FLUX_BURGERS, 0, p) == s
    assert torch.equal(u, ref)


@pytest.mark.parametrize("precision", [0, 1])
def test_step_limit_and_non_finite(npw, precision):
    n = 300
    u0 = _line(n, 1, precision)
    p = npw.Params(precision=precision, max_steps=5)
    ref, st, s = _per_stage(npw, u0, npw.NPW_FLUX_BURGERS, 0, 1.0 / n, 1.0, 0.5, p)
    u = u0.clone()
    with pytest.raises(npw.NpwError) as e:
        npw.npweno_solve(u, 1.0 / n, 1.0, 0.5, npw.NPW_FLUX_BURGERS, 0, p)
    assert e.value.status == npw.NPW_ETIMEOUT == st and s["steps"] == 5 and torch.equal(u, ref)
    u = u0.clone()
    u[0, 123] = float("nan")
    with pytest.raises(npw.NpwError) as e:
        npw.npweno_solve(u, 1.0 / n, 1.0, 0.5, npw.NPW_FLUX_BURGERS, 0, npw.Params(precision=precision))
    assert e.value.status == npw.NPW_ENONFINITE
