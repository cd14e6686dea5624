"""The NPW_FP64 arithmetic with fewer FP64-pipe instructions gives the bits of the plain expressions.

  * Quotients (one reciprocal, Markstein's correction) through the Lax-Friedrichs flux of 1D Euler states:
    bit for bit the flux of numpy float64, whose divisions are correctly rounded, over ordinary densities,
    densities outside the range of the reciprocal (2^-99 .. 2^99), tiny and zero momenta.
  * The monotone switch decided in float with error bounds: on every face, near ties included, the flag of
    the closed form evaluated by numpy float64 in the kernel's order, in FP64 and on float data in the
    mixed path (whose decisions are those of FP64 evaluation); k = 3 variant 0 and the ratio test of k = 2.
  * The near-tie flag decided in float: the same flag as the double expressions give."""
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


def _flux_1d(U, g=1.4):
    rho, mom, E = U
    u = mom / rho
    P = (g - 1.0) * (E - 0.5 * rho * u * u)
    return np.stack([rho * u, rho * u * u + P, (E + P) * u])


@pytest.mark.parametrize("lo,hi,mom", [(0.1, 10.0, 1.0), (1e-3, 1e3, 1e-30), (1e-29, 1e29, 1.0), (1e28, 1e33, 1e20),
                                       (1e-33, 1e-28, 1e-20)])
def test_quotients_are_correctly_rounded(npw, lo, hi, mom):
    g = np.random.default_rng(5)
    n = 200000
    def states():
        rho = np.exp(g.uniform(np.log(lo), np.log(hi), n))
        m = mom * g.normal(size=n)
        m[::97] = 0.0
        return np.stack([rho, m, np.exp(g.uniform(-1, 1, n))])
    a, b = states(), states()
    alpha = 1.7
    with np.errstate(over="ignore", invalid="ignore"):
        ref = 0.5 * (_flux_1d(a) + _flux_1d(b) - alpha * (b - a))
    dev = lambda x: torch.tensor(x, device="cuda")
    h = npw.npweno_flux(dev(a), dev(b), npw.NPW_FLUX_EULER1D, alpha, npw.Params()).cpu().numpy()
    fin = np.isfinite(ref)
    assert np.array_equal(fin, np.isfinite(h))
    assert np.array_equal(h[fin], ref[fin])


def _stencil_data(seed):
    """Smooth, jumps, plateaus, exact steps, round-off noise of several sizes, exact vertex ties."""
    g = np.random.default_rng(seed)
    x = np.arange(4000) / 4000
    u = [1.0 + 0.4 * np.sin(6 * np.pi * x), np.round(8 * np.sin(40 * x)) / 8, np.repeat(g.normal(size=400), 10),
         1.0 + 1e-7 * g.integers(-3, 4, 4000), 1.0 + 2.0 ** -50 * g.integers(-4, 5, 4000), g.normal(size=4000),
         np.cumsum(g.integers(-2, 3, 4000) * 0.25), 1e-3 * (np.arange(4000) % 9) ** 2, g.normal(size=4000) * 1e-25,
         np.repeat([0.0, 1e12, -1e12, 0.0], 1000)]
    return np.concatenate(u)


def _switch_v0(w0, w1, w2, w3):
    A = 6.0 * ((w3 - w0) + 3.0 * (w1 - w2))
    B = 6.0 * ((w0 - w1) + (w3 - w2))
    C = (w0 - w3) + 15.0 * (w2 - w1)
    vm, vp = 4.0 * A - 2.0 * B + C, 4.0 * A + 2.0 * B + C
    mn, mx = np.minimum(vm, vp), np.maximum(vm, vp)
    inside = (A != 0.0) & (np.abs(B) < 4.0 * np.abs(A))
    vv = C - B * B / np.where(A == 0.0, 1.0, 4.0 * A)
    mn, mx = np.where(inside, np.minimum(mn, vv), mn), np.where(inside, np.maximum(mx, vv), mx)
    return (mn < 0.0) & (mx > 0.0)


def _switch_k2(a, b, c):
    num, den = -2.0 * a + 3.0 * b - c, -a + 2.0 * b - c
    r = num / np.where(den == 0.0, 1.0, den)
    return (den != 0.0) & (r > 0.0) & (r < 3.0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("seed", [1, 2])
def test_switch_flags_equal_the_closed_form_everywhere(npw, precision, seed):
    u = _stencil_data(seed)
    if precision:
        u = u.astype(np.float32).astype(np.float64)
    dt = torch.float32 if precision else torch.float64
    n = u.size
    at = lambda k: u[(np.arange(n + 1) + k) % n]  # cell f + k of face f
    d = torch.tensor(u, dtype=dt, device="cuda")
    fl = npw.npweno_reconstruct(d, 0, npw.Params(precision=precision))[2].cpu().numpy()
    assert np.array_equal((fl & 1) != 0, _switch_v0(at(-2), at(-1), at(0), at(1)))
    fl = npw.npweno_reconstruct(d, 0, npw.Params(precision=precision, k=2))[2].cpu().numpy()
    assert np.array_equal((fl & 1) != 0, _switch_k2(at(-2), at(-1), at(0)))
    assert np.array_equal((fl & 8) != 0, _switch_k2(at(-1), at(0), at(1)))


@pytest.mark.parametrize("precision,guard,bound,tol", [(0, 0.0, 0.0, 0.0), (0, 1e-3, 0.05, 1e-6), (1, 0.0, 0.0, 0.0),
                                                       (1, 0.0, 0.3, 1e-5), (0, 0.0, 0.2, 1e-3)])
def test_near_tie_flags_equal_the_double_expressions(npw, precision, guard, bound, tol):
    u = _stencil_data(3)
    if precision:
        u = u.astype(np.float32).astype(np.float64)
    dt = torch.float32 if precision else torch.float64
    n = u.size
    w0, w1, w2, w3 = (u[(np.arange(n + 1) + k) % n] for k in (-2, -1, 0, 1))
    p = npw.Params(precision=precision, eta_guard=guard, eta_max=bound, tie_tol=tol)
    fl = npw.npweno_reconstruct(torch.tensor(u, dtype=dt, device="cuda"), 0, p)[2].cpu().numpy()
    tol = tol or 1e-10
    with np.errstate(all="ignore"):
        A = 6.0 * ((w3 - w0) + 3.0 * (w1 - w2))
        B = 6.0 * ((w0 - w1) + (w3 - w2))
        C = (w0 - w3) + 15.0 * (w2 - w1)
        lim = 12.0 * 8.0 * tol * (np.abs(w0) + np.abs(w1) + np.abs(w2) + np.abs(w3))
        near = (np.abs(4.0 * A - 2.0 * B + C) <= lim) | (np.abs(4.0 * A + 2.0 * B + C) <= lim)
        sv = -B / (2.0 * A)
        v = (A != 0.0) & ((np.abs(np.abs(sv) - 2.0) <= 8.0 * tol) | ((np.abs(sv) < 2.0) & (np.abs(C - B * B / (4.0 * A)) <= lim)))
        near = (near | v) & ~((w0 == w1) & (w1 == w2) & (w2 == w3))
        den = w0 - 15.0 * w1 + 15.0 * w2 - w3
        rel = lambda a, b: (np.maximum(np.abs(a), np.abs(b)) > 0.0) & (np.abs(a - b) <= tol * np.maximum(np.abs(a), np.abs(b)))
        g = guard if guard > 0.0 else (8.0 * 2.0 ** -24 if precision else 0.0)
        if g > 0.0:
            near |= rel(np.abs(den), g * (np.abs(w0) + 15.0 * np.abs(w1) + 15.0 * np.abs(w2) + np.abs(w3)))
        if bound > 0.0:
            near |= rel(np.abs((w0 - 3.0 * w1 + 3.0 * w2 - w3) / (den + 1e-12)), bound)
    assert np.array_equal((fl & 2) != 0, near)
    assert near.any() and not near.all()
