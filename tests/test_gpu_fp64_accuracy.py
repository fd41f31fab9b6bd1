"""The FP64 operator's rounding error against extended precision: the lines run in block fixed point
(fixed.cuh), which may not be less accurate than FP64 arithmetic.

One application of D with a local potential of white noise that dominates it (nothing decays, so
every rounding counts).  Tolerance: six line transforms (three axes, there and back), each with
the statistical error 2^-53 sqrt(log2 W) of an FP64 transform of W points, and four more roundings at
2^-53 (the products with V and the projection), added in quadrature."""
import numpy as np
import pytest

from .test_gpu_work_grid import lib  # noqa: F401  (the fixture)
from .test_gpu_work_grid import _system

pytestmark = pytest.mark.gpu


def _local(ecut, nfft):
    d, x = _system(ecut, nfft, nbnd=2)
    for name in ("beta_kq", "dij"):
        d.pop(name)
    for name in ("kcart", "miller_k", "miller_kq", "u_k", "u_kq", "eps_k"):   # one k-point
        d[name] = d[name][:1]
    d["vloc_r"] = d["vloc_r"] * 1e4
    return d, x[:1]


def _extended(d, x):
    real, cplx = np.longdouble, np.clongdouble
    n, m = d["nfft"], d["miller_kq"][0]
    b = (2 * np.pi * np.linalg.inv(d["lattice"]).T).astype(real)
    g = np.zeros((len(x[0]), n, n, n), cplx)
    g[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n] = x[0]
    r = np.fft.ifftn(g, axes=(1, 2, 3), norm="forward") * d["vloc_r"].astype(real)
    r = np.fft.fftn(r, axes=(1, 2, 3), norm="forward")[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n]
    kin = ((d["kcart"][0].astype(real) + d["q_cart"] + m @ b) ** 2).sum(1) / 2
    t = (kin - d["eps_k"][0].astype(real)[:, None]) * x[0] + r
    u = d["u_kq"][0].astype(cplx)
    return t - (t @ u.conj().T) @ u


@pytest.mark.parametrize("nfft,ecut", [(12, 4.4), (16, 7.9), (24, 17.8), (32, 30.0), (36, 40.0), (48, 50.0), (48, 190.0)])
def test_error_of_an_application(lib, nfft, ecut, monkeypatch):  # noqa: F811
    monkeypatch.setenv("LL_PRUNE", "1")   # transformed on the declared grid
    d, x = _local(ecut, nfft)
    ref = _extended(d, x)
    ch = lib.Chain(approx="rpa", precision="fp64", flavour="nh", max_steps=1, **d)
    err = ch.apply(x, False)[0] - ref
    ch.close()
    rel = float(np.sqrt((abs(err) ** 2).sum() / (abs(ref) ** 2).sum()))
    assert rel <= 2.0 ** -53 * np.sqrt(6 * np.log2(nfft) + 4)


@pytest.mark.parametrize("nfft,ecut", [(16, 7.9), (24, 9.5)])
def test_subnormal_vectors(lib, nfft, ecut, monkeypatch):  # noqa: F811
    """An input whose values are subnormal (2^-1040 of ordinary ones): the operator is linear, and
    each value has 34 bits left, an absolute rounding of 2^-1075 on every one."""
    monkeypatch.setenv("LL_PRUNE", "1")
    d, x = _system(ecut, nfft)
    d.pop("beta_kq")
    d.pop("dij")
    ch = lib.Chain(approx="rpa", precision="fp64", flavour="nh", max_steps=1, **d)
    small = [v.real * 2.0 ** -1040 + 1j * (v.imag * 2.0 ** -1040) for v in x]
    back = [v.real * 2.0 ** 1000 * 2.0 ** 40 + 1j * (v.imag * 2.0 ** 1000 * 2.0 ** 40) for v in small]
    for up in (False, True):
        got = [v.real * 2.0 ** 1000 * 2.0 ** 40 + 1j * (v.imag * 2.0 ** 1000 * 2.0 ** 40) for v in ch.apply(small, up)]
        want = ch.apply(back, up)
        num = sum(np.linalg.norm(p - q) ** 2 for p, q in zip(got, want)) ** 0.5
        assert 0 < num <= 2.0 ** -24 * sum(np.linalg.norm(q) ** 2 for q in want) ** 0.5
    ch.close()
