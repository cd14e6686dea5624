"""The sign of a zero is that of the plain expressions: a face value is a sum from +0, so a field of zeros of
either sign reconstructs to +0; a quotient -0 / rho is -0 and reaches the flux as such."""
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


def _zeros(n, seed):
    return np.where(np.random.default_rng(seed).uniform(size=n) < 0.5, -0.0, 0.0)


@pytest.mark.parametrize("k,precision", [(2, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("scheme", [0, 1, 2, 3])
def test_zero_fields_reconstruct_to_plus_zero(npw, k, precision, scheme):
    u = torch.tensor(_zeros(4001, scheme), dtype=torch.float32 if precision else torch.float64, device="cuda")
    p = npw.Params(k=k, precision=precision, scheme=scheme, eps_M=1e-3)
    vm, vp, _ = npw.npweno_reconstruct(u, 0, p)
    for v in (vm, vp):
        assert (v == 0).all() and not torch.signbit(v).any()


def test_shape_parameter_of_a_zero_numerator(npw):
    # num = ((w0 - 3 w1) + 3 w2) - w3 of zeros is -0 where every term is; eta = num / (den + eps_M)
    w = _zeros(4001, 9)
    at = lambda k: w[(np.arange(4002) + k) % 4001]
    num = ((at(-2) - 3.0 * at(-1)) + 3.0 * at(0)) - at(1)
    eta = npw.npweno_reconstruct(torch.tensor(w, device="cuda"), 0, npw.Params(eps_M=1e-3), True, True)[3].cpu().numpy()
    assert np.signbit(num).any() and (eta == 0).all() and np.array_equal(np.signbit(eta), np.signbit(num))


def test_flux_of_zero_momenta(npw):
    n, g = 3001, np.random.default_rng(2)
    def state():
        return np.stack([g.uniform(0.5, 2.0, n), _zeros(n, g.integers(99)), np.zeros(n)])
    def flux(U):
        rho, m, E = U
        u = m / rho
        P = (1.4 - 1.0) * (E - 0.5 * rho * u * u)
        return np.stack([rho * u, rho * u * u + P, (E + P) * u])
    a, b = state(), state()
    for alpha in (0.0, 1.7):
        ref = 0.5 * (flux(a) + flux(b) - alpha * (b - a))
        h = npw.npweno_flux(torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda"), npw.NPW_FLUX_EULER1D, alpha,
                            npw.Params()).cpu().numpy()
        assert h.tobytes() == ref.tobytes()
