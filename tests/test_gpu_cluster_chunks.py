"""npweno_solve on a short line in launches of 256 steps: runs of several launches give the bits and statistics of
the per-stage kernels (t, dt, alpha, step limit and the float carry go on from one launch to the next), and
the wait limit covers one launch, not the whole solve."""
import time

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
    u = 1.0 + 0.3 * np.sin(2 * np.pi * x + 0.3)
    u = u[None] if m == 1 else np.stack([u, 0.3 * u, 2.0 + u])
    return torch.tensor(u, dtype=torch.float32 if precision else torch.float64, device="cuda")


def _per_stage(npw, u0, kind, bc, dx, t_end, p):
    u = u0.clone()
    m, n = u.shape
    table, _ = npw.make_instances([n], [dx], [t_end], [0.4], [bc], m=m)
    p.batch_mode = 1
    st, stats = npw.npweno_batch_solve(u.reshape(-1), table, m, kind, p, raise_on_error=False)
    return u, st, stats[0]


# steps of advection at speed 1: t_end / (0.4 dx)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,m,bc,steps", [(40, 1, 0, 255), (40, 1, 2, 256), (40, 1, 1, 257), (200, 1, 0, 513), (130, 3, 1, 700)])
def test_runs_of_several_launches(npw, precision, n, m, bc, steps):
    kind = npw.NPW_FLUX_EULER1D if m == 3 else npw.NPW_FLUX_ADVECTION
    u0 = _line(n, m, precision)
    t_end = (steps - 0.5) * 0.4 / n / (1.0 if m == 1 else 1.5)
    p = npw.Params(precision=precision, inflow=(1.1, 0, 0, 0), eta_max=1.0)
    ref, st, s = _per_stage(npw, u0, kind, bc, 1.0 / n, t_end, p)
    assert st == 0 and s["steps"] == steps if m == 1 else s["steps"] > 256
    u = u0.clone()
    assert npw.npweno_solve(u, 1.0 / n, t_end, 0.4, kind, bc, p) == s and torch.equal(u, ref)
    p.max_steps = steps - 3  # the limit in the last launch
    ref, st, s = _per_stage(npw, u0, kind, bc, 1.0 / n, t_end, p)
    u = u0.clone()
    if st == 0:
        assert npw.npweno_solve(u, 1.0 / n, t_end, 0.4, kind, bc, p) == s
    else:
        with pytest.raises(npw.NpwError) as e:
            npw.npweno_solve(u, 1.0 / n, t_end, 0.4, kind, bc, p)
        assert e.value.status == st == npw.NPW_ETIMEOUT
    assert torch.equal(u, ref)


def test_wait_limit_covers_one_launch(npw, monkeypatch):
    n, steps = 1500, 12000
    u = _line(n, 1, 0)
    npw.npweno_solve(u.clone(), 1.0 / n, 0.4 / n, 0.4, npw.NPW_FLUX_ADVECTION, 0, npw.Params())  # load the kernels
    monkeypatch.setenv("NPW_WAIT_TIMEOUT_S", "0.1")
    t0 = time.perf_counter()
    s = npw.npweno_solve(u, 1.0 / n, (steps - 0.5) * 0.4 / n, 0.4, npw.NPW_FLUX_ADVECTION, 0, npw.Params())
    assert s["steps"] == steps and time.perf_counter() - t0 > 0.2
