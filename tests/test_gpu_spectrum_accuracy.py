"""The spectrum of short and weakly damped chains with an extrapolated tail against extended
precision: the device's matrix power over the tail may not be less accurate than the continued
fraction taken row by row in FP64 (NumPy complex128) on the same coefficients (and eight roundings of
the last few operations, which both have)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HA = 27.211386245988


@pytest.fixture(scope="module")
def lib():
    from paper_2111_06623_gb300.build import build_library
    build_library()
    from paper_2111_06623_gb300 import ll
    return ll


def case(m, total, kind, seed):
    rng = np.random.default_rng(seed)
    i = np.arange(m)
    short = lambda v: np.round(v * 2.0 ** 20) / 2.0 ** 20     # sums are exact: one mean in any order
    beta = short(5.6 + 0.3 * (-1.0) ** i + rng.normal(0, 0.02, m))
    gamma = beta * np.exp(1j * rng.normal(0, 0.01, m))
    gamma = short(gamma.real) + 1j * short(gamma.imag)
    z = (rng.normal(size=m) + 1j * rng.normal(size=m)) * np.exp(-i / 30)
    b, g, zz = (np.concatenate([a, np.zeros(total - m, a.dtype)]) for a in (beta, gamma, z))
    h = max(1, m // 2)
    for j in range(m, total):
        pick = slice(h, m) if kind == "constant" else np.arange(h + (h + j) % 2, m, 2)
        b[j], g[j] = beta[pick].mean(), gamma[pick].mean()
    return beta, gamma, z, b, g, zz


def fraction(b, g, z, w, real, cplx):
    b, g, z, w = b.astype(real), g.astype(cplx), z.astype(cplx), w.astype(cplx)
    d, r = w.copy(), np.full(w.shape, z[-1])
    for j in range(len(b) - 2, -1, -1):
        d, r = w - b[j + 1] * g[j + 1] / d, z[j] + b[j + 1] * r / d
    return b[0] * r / d


OMEGA = np.linspace(0.0, 40.0, 101)
CASES = [(64, 100, "osc", 0.1), (64, 400, "osc", 0.1), (64, 3001, "constant", 0.01), (64, 1500, "osc", 0.01)]   # 32 or 16 values a mean


@pytest.mark.parametrize("m,total,kind,eta", CASES)
def test_extrapolated_tail(lib, m, total, kind, eta):
    err, own = 0.0, 0.0
    for seed in (1, 2, 3):
        beta, gamma, z, b, g, zz = case(m, total, kind, seed)
        w = OMEGA / HA + 1j * (eta / HA)
        ref = fraction(b, g, zz, w, np.longdouble, np.clongdouble)
        chi = lib.spectrum(beta, gamma, z, 4.0, [np.sqrt(4 * np.pi), 0, 0], OMEGA, eta, extrapolation=kind, m_total=total)[0]
        rel = lambda v: float((abs(v - ref) ** 2).sum() / (abs(ref) ** 2).sum())
        err += rel(chi)
        own += rel(fraction(b, g, zz, w, np.float64, np.complex128))
    assert err ** 0.5 <= own ** 0.5 + 8 * 2.0 ** -53
