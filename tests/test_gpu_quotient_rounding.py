"""The FP64 quotient is correctly rounded where its reciprocal is hardest: divisors at and just below a power of
two (mantissas of 11 and more leading ones, all ones included), and dividends whose quotient lies as near to a
rounding boundary as any can: 2^k N - X (2 M + 1) = c with c = +-1, +-2, +-3 for the 53-bit mantissas N, X."""
import math
import random

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


def _near_boundaries(X):
    """Mantissas N whose quotient by X is c / (2 X) ulp from a rounding boundary, c small."""
    out = []
    for k in (52, 53, 54):
        for c in (-3, -2, -1, 1, 2, 3):
            m, a, t = 2 * X, 2 ** k, (X + c) % (2 * X)
            g = math.gcd(a, m)
            if t % g:
                continue
            m1 = m // g
            N = (t // g) * pow(a // g, -1, m1) % m1
            N += -(-(2 ** 52 - N) // m1) * m1 if N < 2 ** 52 else 0
            while N < 2 ** 53:
                out.append(N)
                N += m1
    return out


def _check(npw, rho, mom):
    mom = mom * np.where(np.arange(len(mom)) % 2, -1.0, 1.0)
    U = np.stack([rho, mom, np.zeros_like(rho)])
    u = mom / rho
    P = (1.4 - 1.0) * (0.0 - 0.5 * rho * u * u)
    F = np.stack([rho * u, rho * u * u + P, (0.0 + P) * u])
    d = torch.tensor(U, device="cuda")
    h = npw.npweno_flux(d, d.clone(), npw.NPW_FLUX_EULER1D, 0.0, npw.Params()).cpu().numpy()
    assert np.array_equal(h, 0.5 * (F + F)), int((h != 0.5 * (F + F)).any(0).sum())


def test_divisors_below_a_power_of_two(npw):
    r = random.Random(3)
    js = list(range(0, 200)) + [r.randrange(1, 2 ** e) for e in range(8, 53) for _ in range(40)]
    rho, mom = [], []
    for j in js:
        X = 2 ** 53 - max(j, 1)
        for N in _near_boundaries(X) + [2 ** 52, X, 2 ** 53 - 2] + [r.randrange(2 ** 52, 2 ** 53) for _ in range(3)]:
            for s in (0, r.randrange(-60, 60)):
                rho.append(math.ldexp(X, s - 52))
                mom.append(math.ldexp(N, r.randrange(-53, -51)))
    _check(npw, np.array(rho), np.array(mom))


def test_reciprocals_near_a_rounding_boundary(npw):
    """X = 2^53 - j, j odd: 2^105 / X = 2^52 + j / 2 + j^2 2^-54 + .. lies near a boundary where j^2 2^-54 is near an
    integer m."""
    rho, mom = [], []
    for m in range(1, 1500):
        j0 = math.isqrt(m << 54) | 1
        for off in (-900, -300, -100, -30, -8, -2, 0, 2, 8, 30, 100, 300, 900):
            X = 2 ** 53 - (j0 + off)
            for N in _near_boundaries(X):
                rho.append(math.ldexp(X, -52))
                mom.append(math.ldexp(N, -52))
    _check(npw, np.array(rho), np.array(mom))
