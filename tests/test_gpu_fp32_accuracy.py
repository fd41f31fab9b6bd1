"""The rounding error of the FP32 operator: no larger than that of the same transforms with every
twiddled input a product of its own, emulated in NumPy float32.

One application of D with a local potential of white noise that dominates it, on every grid side.
Tolerance: 3% on the ratio of the two rms errors, three times the statistical error of each over
at least 5000 values.  (Butterflies that form a - w b as 2 a - (a + w b) are 3 to 14% over.)"""
import numpy as np
import pytest

from .test_gpu_work_grid import lib  # noqa: F401  (the fixture)
from .test_gpu_work_grid import _system

pytestmark = pytest.mark.gpu

F, D = np.float32, np.float64
PLAN = {12: (4, 3), 16: (4, 4), 18: (3, 3, 2), 24: (4, 3, 2), 32: (4, 4, 2), 36: (4, 3, 3), 48: (4, 4, 3)}


def fma(a, b, c):      # float32 fused multiply-add (the product is exact in float64)
    return (a.astype(D) * D(b) + c).astype(F) if np.ndim(b) == 0 else (a.astype(D) * b + c).astype(F)


def mul(a, w):         # complex product, pairs (re, im)
    return fma(a[0], w[0], (-a[1] * w[1]).astype(F)), fma(a[0], w[1], (a[1] * w[0]).astype(F))


def add(a, b):
    return a[0] + b[0], a[1] + b[1]


def sub(a, b):
    return a[0] - b[0], a[1] - b[1]


def turn(a, s):        # s i a
    return (-a[1], a[0]) if s > 0 else (a[1], -a[0])


def dft(v, s):
    if len(v) == 2:
        return [add(v[0], v[1]), sub(v[0], v[1])]
    if len(v) == 3:
        t, d = add(v[1], v[2]), sub(v[1], v[2])
        c = F(s * 0.8660254037844386)
        m = fma(t[0], F(-0.5), v[0][0]), fma(t[1], F(-0.5), v[0][1])
        return [add(v[0], t), (fma(d[1], -c, m[0]), fma(d[0], c, m[1])), (fma(d[1], c, m[0]), fma(d[0], -c, m[1]))]
    a, b, c, d = add(v[0], v[2]), sub(v[0], v[2]), add(v[1], v[3]), turn(sub(v[1], v[3]), s)
    return [add(a, c), add(b, d), sub(a, c), sub(b, d)]


def transform(x, s, axis):
    """Unnormalised float32 transform of the pair of arrays x along an axis."""
    n = x[0].shape[axis]
    a = [tuple(np.take(p, i, axis) for p in x) for i in range(n)]
    ns = 1
    for r in PLAN[n]:
        out = [None] * n
        for j in range(n // r):
            v = []
            for q in range(r):
                e = (j % ns) * q * (n // (ns * r))
                w = np.exp(s * 2j * np.pi * e / n)
                v.append(mul(a[j + q * (n // r)], (F(w.real), F(w.imag))) if e else a[j + q * (n // r)])
            for q, o in enumerate(dft(v, s)):
                out[(j // ns) * ns * r + j % ns + q * ns] = o
        a, ns = out, ns * r
    return tuple(np.stack([p[c] for p in a], axis) for c in (0, 1))


def emulated(d, k, x):
    n, m = d["nfft"], d["miller_kq"][k]
    g = np.zeros((len(x), n, n, n), complex)
    g[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n] = x
    g = g.real.astype(F), g.imag.astype(F)
    for axis in (3, 1, 2):
        g = transform(g, +1, axis)
    v = d["vloc_r"].astype(F)
    g = g[0] * v, g[1] * v
    for axis in (2, 1, 3):
        g = transform(g, -1, axis)
    sel = (slice(None), m[:, 0] % n, m[:, 1] % n, m[:, 2] % n)
    t = tuple((p[sel] * F(1 / n ** 3)).astype(F) for p in g)
    b = 2 * np.pi * np.linalg.inv(d["lattice"]).T
    kin = (0.5 * ((d["kcart"][k] + d["q_cart"] + m @ b) ** 2).sum(1)[None] - d["eps_k"][k][:, None]).astype(F)
    t = fma(x.real.astype(F), kin, t[0]), fma(x.imag.astype(F), kin, t[1])
    for u, c in zip(d["u_kq"][k], ((t[0] + 1j * t[1]).astype(complex) @ d["u_kq"][k].conj().T).T):   # P_c
        for v in range(len(x)):
            p = mul((u.real.astype(F), u.imag.astype(F)), (F(c[v].real), F(c[v].imag)))
            t[0][v], t[1][v] = t[0][v] - p[0], t[1][v] - p[1]
    return t[0].astype(D) + 1j * t[1]


def exact(d, k, x):
    n, m = d["nfft"], d["miller_kq"][k]
    g = np.zeros((len(x), n, n, n), complex)
    g[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n] = x
    r = np.fft.fftn(np.fft.ifftn(g, axes=(1, 2, 3)) * d["vloc_r"], axes=(1, 2, 3))
    b = 2 * np.pi * np.linalg.inv(d["lattice"]).T
    kin = 0.5 * ((d["kcart"][k] + d["q_cart"] + m @ b) ** 2).sum(1)[None] - d["eps_k"][k][:, None]
    t = kin * x + r[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n]
    return t - (t @ d["u_kq"][k].conj().T) @ d["u_kq"][k]


@pytest.mark.parametrize("nfft,ecut,nbnd", [(12, 9.0, 8), (16, 24.0, 8), (18, 26.0, 8), (24, 17.8, 8), (32, 30.0, 3),
                                            (36, 40.0, 3), (48, 50.0, 2)])
def test_error_of_an_application(lib, nfft, ecut, nbnd, monkeypatch):  # noqa: F811
    monkeypatch.setenv("LL_PRUNE", "1")   # transformed on the declared grid
    d, x = _system(ecut, nfft, nbnd=nbnd)
    for name in ("beta_kq", "dij"):
        d.pop(name)
    d["vloc_r"] = (d["vloc_r"] * 1e4).astype(F).astype(D)      # inputs that FP32 holds
    d["u_kq"] = [u.astype(np.complex64).astype(complex) for u in d["u_kq"]]
    x = [v.astype(np.complex64).astype(complex) for v in x]
    assert sum(v.size for v in x) >= 5000
    ch = lib.Chain(approx="rpa", precision="fp32", flavour="nh", max_steps=1, **d)
    got = ch.apply(x, False)
    ch.close()
    ref = [exact(d, k, v) for k, v in enumerate(x)]
    own = sum((abs(emulated(d, k, v) - r) ** 2).sum() for k, (v, r) in enumerate(zip(x, ref))) ** 0.5
    err = sum((abs(g - r) ** 2).sum() for g, r in zip(got, ref)) ** 0.5
    print("rms error %.3g of the result, emulated %.3g" % tuple(v / sum((abs(r) ** 2).sum() for r in ref) ** 0.5 for v in (err, own)))
    assert err <= 1.03 * own
