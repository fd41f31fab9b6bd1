"""The FP32 plane pass and the per-k paths on every grid side, bound and lane split, against NumPy:
the counterpart of the FP64 applications of test_gpu_fixed_lines.py (whose 48-point lines, and
whose density pass at 32, run on lane pairs in FP32 too), and the tensor-core projections beside
them.  Tolerance 2e-5 of the output's norm, as in the FP32 oracle parity tests."""
import numpy as np
import pytest

from .test_gpu_fixed_lines import GRIDS, _reference
from .test_gpu_work_grid import _system, lib  # noqa: F401  (lib: the fixture)

pytestmark = pytest.mark.gpu


def _with_projectors(d, x, upper):
    """(D + K) x of a system with Kleinman-Bylander projectors."""
    bare = _reference(d, x, upper)
    out = []
    for t, v, b, u in zip(bare, x, d["beta_kq"], d["u_kq"]):
        kb = (v @ b.conj().T * d["dij"]) @ b
        out.append(t + kb - (kb @ u.conj().T) @ u)
    return out


def _check(got, ref, tol=2e-5):
    num = sum(np.linalg.norm(p - q) ** 2 for p, q in zip(got, ref)) ** 0.5
    assert num <= tol * sum(np.linalg.norm(q) ** 2 for q in ref) ** 0.5


@pytest.mark.parametrize("nfft,ecut", GRIDS)
def test_fp32_application(lib, nfft, ecut, monkeypatch):  # noqa: F811
    monkeypatch.setenv("LL_PRUNE", "1")   # transformed on the declared grid
    d, x = _system(ecut, nfft)
    ch = lib.Chain(approx="rpa", precision="fp32", max_steps=1, flavour="nh", **d)
    for upper in (False, True):
        _check(ch.apply(x, upper), _with_projectors(d, x, upper))
    ch.close()


@pytest.mark.parametrize("nfft,ecut", [(16, 7.9), (32, 20.0), (48, 50.0), (48, 135.0)])
def test_fp32_application_with_tensor_core_projections(lib, nfft, ecut, monkeypatch):  # noqa: F811
    monkeypatch.setenv("LL_PRUNE", "1")
    monkeypatch.setenv("LL_SPLIT_PERK", "1")
    d, x = _system(ecut, nfft, nbnd=8, nproj=12)
    ch = lib.Chain(approx="rpa", precision="fp32", max_steps=1, flavour="nh", **d)
    for upper in (False, True):
        _check(ch.apply(x, upper), _with_projectors(d, x, upper))
    ch.close()


# side, cut-off, largest |m|: one beyond side/4, at side/4 + 2 and one beyond (the bounds of the lines)
BOUNDS = [(24, 37.0, 7), (24, 48.0, 8), (24, 61.0, 9), (32, 61.0, 9), (32, 75.0, 10), (32, 91.0, 11), (36, 75.0, 10), (36, 90.0, 11),
          (36, 108.0, 12), (48, 127.0, 13), (48, 147.0, 14), (48, 170.0, 15)]


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
@pytest.mark.parametrize("nfft,ecut,mmax", BOUNDS)
def test_line_bounds(lib, nfft, ecut, mmax, precision, tol, monkeypatch):  # noqa: F811
    monkeypatch.setenv("LL_PRUNE", "1")
    d, x = _system(ecut, nfft, nbnd=2)
    assert max(abs(m).max() for m in d["miller_kq"]) == mmax
    ch = lib.Chain(approx="rpa", precision=precision, max_steps=1, flavour="nh", **d)
    for upper in (False, True):
        _check(ch.apply(x, upper), _with_projectors(d, x, upper), tol)
    ch.close()


# bands, copies of the eight k-points: groups of 1, 2 (and 4 bands of the non-Hermitian update), 3 and 4
# bands per CTA, and the bands that blocks of two and four leave over
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
@pytest.mark.parametrize("nbnd,copies", [(1, 1), (2, 1), (3, 1), (5, 24), (6, 8), (9, 8), (12, 8), (13, 24)])
def test_band_groups(lib, nbnd, copies, precision, tol):  # noqa: F811
    for nproj in (1, 2, 6):
        d, x = _system(5.5, 12, nbnd=nbnd, nproj=nproj)
        for name in ("miller_k", "miller_kq", "u_k", "u_kq", "beta_kq"):
            d[name] = d[name] * copies
        d["kcart"], d["eps_k"] = (np.tile(d[name], (copies, 1)) for name in ("kcart", "eps_k"))
        rng = np.random.default_rng(nbnd)
        x = [v * rng.normal() for v in x * copies]
        ch = lib.Chain(approx="rpa", precision=precision, max_steps=1, flavour="nh", **d)
        for upper in (False, True):
            _check(ch.apply(x, upper), _with_projectors(d, x, upper), tol)
        ch.close()
