"""Orbitals transformed on a smaller grid than the declared one where the spheres' differences
fit it (chain.cuh, work_side): one application against the same system on the declared grid
(LL_PRUNE=1), over every pair of sides, options and Q that take it, at the single-application
tolerances of the oracle parity tests (1e-12 in FP64, 2e-5 in FP32: the same sums, other
rounding); and the device bytes, which show that the smaller grid was taken, or was not."""
import numpy as np
import pytest

import workloads as w
from workloads.cells import grid_operations, irreducible_kpoints, kmesh_frac, small_group, sphere

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2111_06623_gb300.build import build_library
    build_library()
    from paper_2111_06623_gb300 import ll
    return ll


def _system(ecut, nfft, q=(0.1, 0.0, 0.0), nbnd=3, nproj=2, wedge=False, metal=False, ecut_q=None, seed=3):
    """A random system on the two-atom cell: orthonormal orbitals, smooth positive density."""
    spec = w.config_small()
    spec.ecut_ry, spec.nfft, spec.kmesh = ecut, nfft, (2, 2, 2)
    spec.q_cart = np.asarray(q) * (2 * np.pi / w.A_LAT)
    rng = np.random.default_rng(seed)
    b = spec.bvec
    kf, d = kmesh_frac(spec.kmesh), {}
    if wedge:
        ops = small_group(spec)
        kf, d["kweight"] = irreducible_kpoints(spec, ops)
        d["sym"] = grid_operations(spec, ops)
        assert len(ops) > 1
    kc = kf @ b
    mk = [sphere(k, b, ecut) for k in kc]
    mq = [sphere(k + spec.q_cart, b, ecut_q or ecut) for k in kc]

    def states(m, n):
        x = rng.normal(size=(len(m), n)) + 1j * rng.normal(size=(len(m), n))
        return np.linalg.qr(x)[0].T.copy()

    n = nfft
    r = np.indices((n, n, n)) * (2 * np.pi / n)
    rho = 0.02 + 0.01 * np.cos(r[0]) * np.cos(r[1] - r[2])
    if wedge:
        j = np.indices((n, n, n)).reshape(3, -1)
        rho = np.mean([rho[tuple((s @ j) % n)] for s in d["sym"]], axis=0).reshape(n, n, n)
    if metal:
        nk = len(kc)
        d.update(occ_k=rng.uniform(0.5, 1, (nk, nbnd)), occ_kq=rng.uniform(0, 1, (nk, nbnd)),
                 eps_kq=rng.normal(size=(nk, nbnd)))
    d.update(lattice=spec.lattice, nfft=n, kcart=kc, miller_k=mk, miller_kq=mq, u_k=[states(m, nbnd) for m in mk],
             u_kq=[states(m, nbnd) for m in mq], eps_k=rng.normal(size=(len(kc), nbnd)) - 9.0,
             vloc_r=rng.normal(size=(n, n, n)), rho_r=rho, q_cart=spec.q_cart,
             beta_kq=[rng.normal(size=(nproj, len(m))) + 1j * rng.normal(size=(nproj, len(m))) for m in mq],
             dij=rng.normal(size=nproj))
    x = [rng.normal(size=(nbnd, len(m))) + 1j * rng.normal(size=(nbnd, len(m))) for m in mq]
    return d, x


# (ecut, declared side, extra, smaller grid expected)
CASES = {
    "18->16": (10.0, 18, {}, True),
    "16->12": (4.0, 16, {}, True),
    "18->12": (4.0, 18, {}, True),
    "24->16": (10.0, 24, {}, True),
    "32->24": (25.0, 32, {}, True),
    "36->32": (38.0, 36, {}, True),
    "48->36": (52.0, 48, {}, True),
    "48->12": (4.0, 48, {}, True),
    "same": (5.5, 12, {}, False),
    "tight": (16.0, 24, {}, False),
    "beyond the zone": (10.0, 18, dict(q=(1.3, 0.2, 0.1)), True),
    "far beyond": (4.0, 16, dict(q=(4.0, 0.2, 0.1)), False),
    "other cut-off at k+Q": (10.0, 32, dict(ecut_q=22.0), True),
    "wedge": (10.0, 24, dict(wedge=True), True),
    "metal": (10.0, 18, dict(metal=True), True),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
def test_work_grid_matches_declared_grid(lib, name, precision, tol, monkeypatch):
    ecut, n, extra, smaller = CASES[name]
    d, x = _system(ecut, n, **extra)
    for approx in ("tddft", "rpa"):
        got, size = {}, {}
        for env in ("1", ""):
            monkeypatch.setenv("LL_PRUNE", env)
            ch = lib.Chain(precision=precision, flavour="nh", approx=approx, max_steps=4, **d)
            got[env] = [ch.apply(x, up) for up in (True, False)]
            size[env] = ch.bytes()
            ch.close()
        assert (size[""] < size["1"]) == smaller
        for a, b in zip(got[""], got["1"]):
            scale = max(np.max(np.abs(v)) for v in b)
            assert max(np.max(np.abs(u - v)) for u, v in zip(a, b)) <= tol * scale
