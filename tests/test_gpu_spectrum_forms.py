"""The division-free elimination of the spectrum kernel and its matrix power over the extrapolated
tail, against the division form of the continued fraction in NumPy complex128, at the lengths
where the row blocks (32, scaled every 4), the period-two tail and the frequency blocks have
edges.  Tolerance 1e-10 relative to the largest value, the device spectrum's tolerance against
the oracle: both forms are backward recursions whose rounding errors stay near 1e-14."""
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


def _division_form(beta, gamma, z, w, eta):
    wc = (w + 1j * eta) / HA
    d, r = wc.copy(), np.full(wc.shape, z[-1])
    for j in range(len(beta) - 2, -1, -1):
        d, r = wc - beta[j + 1] * gamma[j + 1] / d, z[j] + beta[j + 1] * r / d
    return beta[0] * r / d


@pytest.mark.parametrize("m,extra", [(1, 0), (2, 0), (5, 0), (33, 0), (34, 0), (65, 0), (1000, 0), (4, 1), (4, 2),
                                     (5, 1), (64, 3), (97, 4096), (98, 19903), (1000, 19000)])
@pytest.mark.parametrize("kind", ["constant", "osc"])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e30])
def test_spectrum_rows_and_tail(lib, m, extra, kind, scale):
    if extra and m < (4 if kind == "osc" else 2):
        pytest.skip("too few coefficients to extrapolate")
    rng = np.random.default_rng(m + extra)
    i = np.arange(m)
    beta = scale * (5.0 + 0.5 * (-1.0) ** i + rng.normal(0, 0.05, m))
    gamma = beta * np.exp(1j * rng.normal(0, 0.02, m))
    z = rng.normal(size=m) + 1j * rng.normal(size=m)
    w, eta = scale * np.linspace(0.0, 300.0, 67), scale * 0.5
    b, g, zz = (np.concatenate([a, np.zeros(extra, a.dtype)]) for a in (beta, gamma, z))
    h = max(1, m // 2)
    for j in range(m, m + extra):
        pick = slice(h, m) if kind == "constant" else np.arange(h + (h + j) % 2, m, 2)
        b[j], g[j] = beta[pick].mean(), gamma[pick].mean()
    ref = _division_form(b, g, zz, w, eta)
    chi, ei, e = lib.spectrum(beta, gamma, z, 4.0, [np.sqrt(4 * np.pi), 0, 0], w, eta,
                              extrapolation=kind if extra else "no", m_total=m + extra)
    assert np.max(np.abs(chi - ref)) <= 1e-10 * np.max(np.abs(ref))
    assert np.max(np.abs(ei - 1 - ref)) <= 1e-10 * np.max(np.abs(1 + ref))
    assert np.max(np.abs(e * ei - 1)) <= 1e-10
