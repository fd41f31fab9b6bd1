"""Spheres at k+Q beyond half the grid (a Q far outside the first zone): indexed from a reciprocal
lattice vector of their own where that brings them within the plane pass's range (chain.cuh,
fold_index), on the general plane kernel (k_xy) where it does not; and spheres that fill the grid.
Single applications against NumPy on the declared grid, at the tolerances of the oracle parity tests
(1e-12 in FP64, 2e-5 in FP32)."""
import numpy as np
import pytest

from .test_gpu_sides import _check, _with_projectors
from .test_gpu_work_grid import _system, lib  # noqa: F401  (lib: the fixture)

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-5}

# side, cut-off, Q along x (2 pi / a): spheres at k+Q beyond half the grid; the second beyond the grid itself
FAR = [(12, 9.0, 8.0), (18, 51.84, 21.8), (16, 20.0, 8.0), (18, 20.0, 11.0), (24, 38.0, 13.0), (32, 55.0, 18.0), (36, 70.0, 22.0),
       (48, 110.0, 28.0)]
# side, cut-off, Q: the spheres fill the grid and are not all in one range of its side
WIDE = [(12, 25.056, (0.9, 0.4, 0.2)), (16, 45.568, (0.9, 0.4, 0.2)), (24, 103.68, (0.9, 0.4, 0.2)), (32, 186.368, (0.9, 0.4, 0.2)),
        (48, 423.936, (0.9, 0.4, 0.2))]


def _apply(lib, d, x, precision, flavour="nh", **kw):  # noqa: F811
    ch = lib.Chain(approx="rpa", precision=precision, flavour=flavour, max_steps=4, **d, **kw)
    out = [ch.apply(x, up) for up in (False, True)]
    ch.close()
    return out


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nfft,ecut,q", FAR)
def test_far_q(lib, nfft, ecut, q, precision):  # noqa: F811
    d, x = _system(ecut, nfft, q=(q, 0.2, 0.1))
    assert max(abs(m).max() for m in d["miller_kq"]) > (nfft if q == 21.8 else nfft // 2)
    for up, got in enumerate(_apply(lib, d, x, precision)):
        _check(got, _with_projectors(d, x, up), TOL[precision])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nfft,ecut,q", WIDE)
def test_spheres_that_fill_the_grid(lib, nfft, ecut, q, precision):  # noqa: F811
    d, x = _system(ecut, nfft, q=q, nbnd=2)
    lo, hi = (np.array([f(m, axis=0) for m in d["miller_kq"]]) for f in (np.min, np.max))
    assert (hi - lo).max() < nfft <= (hi.max(0) - lo.min(0)).max()
    for up, got in enumerate(_apply(lib, d, x, precision)):
        _check(got, _with_projectors(d, x, up), TOL[precision])


def zones(d):
    """Some of the k-points given in other zones: no one index shift fits the spheres."""
    n, b = d["nfft"], 2 * np.pi * np.linalg.inv(d["lattice"]).T
    d["kcart"] = d["kcart"].copy()
    for k in (1, 4, 6):
        g = np.array([n, -n // 2, 3])
        d["kcart"][k] += g @ b
        for name in ("miller_k", "miller_kq"):
            d[name][k] = d[name][k] - g


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nfft,ecut", [(12, 4.4), (18, 10.0), (24, 17.8), (32, 20.0), (36, 40.0), (48, 50.0)])
def test_k_points_in_different_zones(lib, nfft, ecut, precision):  # noqa: F811
    """The general plane kernel (k_xy)."""
    d, x = _system(ecut, nfft, nbnd=2)
    zones(d)
    for up, got in enumerate(_apply(lib, d, x, precision)):
        _check(got, _with_projectors(d, x, up), TOL[precision])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_k_points_beyond_the_grid(lib, precision):  # noqa: F811
    """k given a reciprocal lattice vector outside the zone: both families of spheres move."""
    d, x = _system(10.0, 18)
    g = np.array([-25, 3, -40])
    d["kcart"] = d["kcart"] + g @ (2 * np.pi * np.linalg.inv(d["lattice"]).T)
    for name in ("miller_k", "miller_kq"):
        d[name] = [m - g for m in d[name]]
    for up, got in enumerate(_apply(lib, d, x, precision)):
        _check(got, _with_projectors(d, x, up), TOL[precision])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_far_q_on_a_wedge(lib, precision, monkeypatch):  # noqa: F811
    """The wedge of the small group against the same chain on the declared grid, f_xc included."""
    d, x = _system(38.0, 24, q=(13.0, 0.0, 0.0), wedge=True)
    assert max(abs(m).max() for m in d["miller_kq"]) > 12
    out = []
    for env in ("", "1"):
        monkeypatch.setenv("LL_PRUNE", env)
        ch = lib.Chain(precision=precision, flavour="nh", max_steps=4, **d)
        out.append(ch.apply(x, True))
        ch.close()
    _check(out[0], out[1], TOL[precision])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_far_q_shares_the_ground_states_grids(lib, precision):  # noqa: F811
    near, _ = _system(20.0, 16)
    far, _ = _system(20.0, 16, q=(8.0, 0.2, 0.1))
    for name in ("u_k", "eps_k", "vloc_r", "rho_r"):
        far[name] = near[name]
    kw = dict(precision=precision, flavour="nh", max_steps=6)
    lender, own = lib.Chain(**kw, **near), lib.Chain(**kw, **far)
    shared = lib.Chain(share=lender, **kw, **far)
    assert shared.bytes() < own.bytes()
    for a, b in zip(shared.lanczos(6), own.lanczos(6)):
        assert np.array_equal(a, b)
