"""ll_apply pads and unpads the caller's packed vector on the device: FP32 and FP64, the packed
vector within the column buffer and (FP32, spheres that fill the grid) beyond it; the non-Hermitian
chain (two vectors of columns) too; against NumPy, list and packed inputs alike.

Tolerances: those of the single-application oracle tests, 1e-12 in FP64 and 2e-5 in FP32."""
import numpy as np
import pytest

from .test_gpu_fixed_lines import _reference
from .test_gpu_work_grid import _system, lib  # noqa: F401  (lib: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
@pytest.mark.parametrize("nfft,ecut", [(18, 10.0), (24, 95.0)])
@pytest.mark.parametrize("flavour", ["ph", "nh"])
def test_packed(lib, nfft, ecut, precision, tol, flavour, monkeypatch):  # noqa: F811
    monkeypatch.setenv("LL_PRUNE", "1")
    d, x = _system(ecut, nfft)
    d.pop("beta_kq")
    d.pop("dij")
    if nfft == 24:   # the packed vector (16 bytes a value) against FP32 columns, one vector
        cols = max(len(np.unique(m[:, :2], axis=0)) for m in d["miller_k"] + d["miller_kq"])
        assert 8 * len(x) * nfft * (cols + cols % 2) < 16 * sum(len(m) for m in d["miller_kq"])
    ch = lib.Chain(approx="rpa", flavour=flavour, precision=precision, max_steps=1, **d)
    flat = np.concatenate([v.ravel() for v in x])
    for upper in (False, True):
        ref = _reference(d, x, upper)
        got = ch.apply(flat, upper)
        num = sum(np.linalg.norm(p - q) ** 2 for p, q in zip(got, ref)) ** 0.5
        assert num <= tol * sum(np.linalg.norm(q) ** 2 for q in ref) ** 0.5
        for p, q in zip(ch.apply(x, upper), got):
            assert np.array_equal(p, q)
    ch.close()
