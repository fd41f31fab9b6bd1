"""The FP64 plane pass in 64-bit block fixed point (fixed.cuh, plane64.cuh): one application on
every grid side and pruning level, with and without the response potential, against NumPy; inputs
of any magnitude, of uneven magnitudes, zero and not finite.

Tolerance: 1e-12 of the output's norm, as in the FP64 oracle parity tests (a line rounds at 2^-53
of its largest value or below, and a vector's lines are at most its norm)."""
import numpy as np
import pytest

from .test_gpu_work_grid import _system, lib  # noqa: F401  (lib: the fixture)

pytestmark = pytest.mark.gpu

# (declared side, cut-off): the spheres at |m| <= side/4, at side/2 - 1 (48 also at 14)
GRIDS = [(12, 4.4), (12, 13.0), (16, 7.9), (16, 24.0), (18, 10.0), (18, 26.0), (24, 9.5), (24, 50.0), (32, 20.0), (32, 85.0),
         (36, 40.0), (36, 100.0), (48, 50.0), (48, 135.0), (48, 190.0)]


def _reference(d, x, upper):
    """(D + K) x (RPA) in NumPy; K without the exchange-correlation kernel."""
    n, lat = d["nfft"], d["lattice"]
    b = 2 * np.pi * np.linalg.inv(lat).T
    om = abs(np.linalg.det(lat))
    grid = lambda c, m: np.fft.ifftn(_box(c, m, n), axes=(1, 2, 3), norm="forward")
    t, dens = [], np.zeros((n, n, n), complex)
    for k, m in enumerate(d["miller_kq"]):
        r = grid(x[k], m)
        kin = 0.5 * ((d["kcart"][k] + d["q_cart"] + m @ b) ** 2).sum(1)
        t.append((kin - d["eps_k"][k][:, None]) * x[k] + _pick(r * d["vloc_r"], m))
        dens += (grid(d["u_k"][k], d["miller_k"][k]).conj() * r).sum(0)
    if upper:
        f = np.fft.fftfreq(n, 1 / n)
        g = np.stack(np.meshgrid(f, f, f, indexing="ij"), -1) @ b + d["q_cart"]
        vp = np.fft.ifftn(np.fft.fftn(4 / (om * len(t)) * dens) * 4 * np.pi / (g * g).sum(-1))
        for k, m in enumerate(d["miller_kq"]):
            t[k] = t[k] + _pick(grid(d["u_k"][k], d["miller_k"][k]) * vp, m)
    return [v - (v @ u.conj().T) @ u for v, u in zip(t, d["u_kq"])]


def _box(c, m, n):
    out = np.zeros((len(c), n, n, n), complex)
    out[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n] = c
    return out


def _pick(r, m):
    n = r.shape[-1]
    return np.fft.fftn(r, axes=(1, 2, 3), norm="forward")[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n]


def _open(lib, nfft, ecut, monkeypatch):  # noqa: F811
    monkeypatch.setenv("LL_PRUNE", "1")   # transformed on the declared grid
    d, x = _system(ecut, nfft)
    d.pop("beta_kq")
    d.pop("dij")
    return d, x, lib.Chain(approx="rpa", precision="fp64", max_steps=1, **d)


def _close(a, b):
    num = sum(np.linalg.norm(p - q) ** 2 for p, q in zip(a, b)) ** 0.5
    assert num <= 1e-12 * sum(np.linalg.norm(q) ** 2 for q in b) ** 0.5


@pytest.mark.parametrize("nfft,ecut", GRIDS)
@pytest.mark.parametrize("upper", [False, True])
def test_application(lib, nfft, ecut, upper, monkeypatch):  # noqa: F811
    d, x, ch = _open(lib, nfft, ecut, monkeypatch)
    ref = _reference(d, x, upper)
    _close(ch.apply(np.concatenate([v.ravel() for v in x]), upper), ref)
    rng = np.random.default_rng(5)      # components over twelve decades
    x = [v * 10.0 ** rng.uniform(-12, 0, v.shape) for v in x]
    _close(ch.apply(np.concatenate([v.ravel() for v in x]), upper), _reference(d, x, upper))
    ch.close()


@pytest.mark.parametrize("nfft,ecut", [(16, 7.9), (24, 9.5)])
def test_magnitudes(lib, nfft, ecut, monkeypatch):  # noqa: F811
    d, x, ch = _open(lib, nfft, ecut, monkeypatch)
    flat = np.concatenate([v.ravel() for v in x])
    ref = ch.apply(flat, True)
    for s in (2.0 ** -700, 2.0 ** 700):
        _close([v / s for v in ch.apply(flat * s, True)], ref)
    assert all((v == 0).all() for v in ch.apply(0 * flat, True))
    ref = ch.apply(flat, False)
    for bad in (np.nan, np.inf):        # an orbital with a value that is not finite: itself, no other
        y = flat.copy()
        y[7] = bad
        out = ch.apply(y, False)
        assert not np.isfinite(out[0][0]).any()
        assert np.array_equal(out[0][1:], ref[0][1:]) and all(np.array_equal(p, q) for p, q in zip(out[1:], ref[1:]))
    ch.close()
