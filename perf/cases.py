"""The work a user of the Liouville-Lanczos library has it do, as measurable cases.

A case is one of three kinds of call through the public binding (`paper_2111_06623_gb300.ll`):

  chain     n more Lanczos steps of a resident chain (`Chain.lanczos`), the library's main path:
            every pass continues the chain, as a program that runs a recursion in portions (and
            the request loop) does; a chain that has reached its 5000 steps (the number of
            iterations the method is run to without extrapolation) is followed by a new one of
            the same system.  Outputs: every coefficient so far.
  apply     one application of the operator to a batch of host vectors (`Chain.apply`), the
            building block of a program with an iteration of its own.  Outputs: the batch.
  spectrum  chi, eps^-1 and eps of caller-held coefficients on a frequency grid, extrapolated
            (`ll.spectrum`), the post-processing of a finished chain.

The crystals are the repository's: the two-atom FCC diamond cell (a = 10.26 bohr), its
eight-atom cubic cell and its sixteen-atom supercell, with the cut-offs, grids, k-meshes, bands
and projectors of its configurations and tests.  A ground state is a model of the real one that
takes milliseconds: the ions' smeared Coulomb wells screened by a valence density of Gaussian
bond orbitals, those orbitals orthonormalised at every k and k+Q, band energies below the
spectrum of the Hamiltonian on the empty states (an insulator: D is positive).  The metal's
states and levels are the eigenstates of its Hamiltonian, its density theirs.

Results of an FP32 chain are kept in 32 bits, as they carry no more.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_2111_06623_gb300 import ll

A = 10.26                 # bohr, the lattice parameter of every cell
MAX_STEPS = 5000          # capacity of a chain
HA_EV = 27.211386245988


# ---- the listed cases -------------------------------------------------------------------
def _case(name=None, kind="chain", cell="fcc", ecut=10.0, nfft=18, k1=4, k2=4, k3=4, nbnd=4, per_atom=1, prec="fp32",
          flavour="ph", approx="tddft", q=0.1, steps=10, stream=True, wedge=False, metal=False):
    c = dict(kind=kind, cell=cell, ecut=ecut, nfft=nfft, k1=k1, k2=k2, k3=k3, nbnd=nbnd, per_atom=per_atom, prec=prec,
             flavour=flavour, approx=approx, q=q, steps=steps, stream=stream, wedge=wedge, metal=metal)
    return dict(name=name, **c) if name else c


def _spectrum_case(name=None, m=1000, m_total=20000, n_omega=4001, extrap="osc"):
    c = dict(kind="spectrum", m=m, m_total=m_total, n_omega=n_omega, extrap=extrap)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest cell (4 Ry, 12^3, 8 k-points) on the default stream: latency and launches
        _case("tiny_fp64", ecut=4.0, nfft=12, k1=2, k2=2, k3=2, prec="fp64", steps=20, stream=False),
        # the plain method: two-atom cell, 10 Ry, 18^3, 64 k-points, FP64, a first script's default stream
        _case("small_fp64", prec="fp64", steps=20, stream=False),
        # one chain of a many-Q sweep on that cell: FP32, larger Q, its own stream
        _case("small_fp32", q=0.45),
        # the semimetal: smeared occupations, 6 bands
        _case("metal_fp32", nbnd=6, per_atom=0, metal=True),
        # the benchmark's workload: KB s/p projectors, 25 Ry, 32^3, 512 k-points, both precisions
        _case("kb_fp32", ecut=25.0, nfft=32, k1=8, k2=8, k3=8, per_atom=4),
        _case("kb_fp64", ecut=25.0, nfft=32, k1=8, k2=8, k3=8, per_atom=4, prec="fp64"),
        # ... its non-Hermitian recursion (two applications per step)
        _case("kb_nh_fp32", ecut=25.0, nfft=32, k1=8, k2=8, k3=8, per_atom=4, flavour="nh", steps=5),
        # ... and its irreducible wedge under the small group of Q (ragged: 164 k-points with weights)
        _case("kb_wedge_fp32", ecut=25.0, nfft=32, k1=8, k2=8, k3=8, per_atom=4, wedge=True),
        # eight-atom cubic cell: 16 bands, ~1630 plane waves, band groups per CTA
        _case("cubic8_fp32", cell="cubic", ecut=20.0, nfft=32, nbnd=16, per_atom=1),
        # sixteen-atom supercell: 32 bands, 64 projectors, ~6000 plane waves, 48^3: the largest
        _case("sc16_fp32", cell="super", ecut=30.0, nfft=48, nbnd=32, per_atom=4, q=0.15, steps=6),
        # one application of the eight-atom cell's operator to host vectors, FP64
        _case("apply_cubic8_fp64", kind="apply", cell="cubic", ecut=20.0, nfft=32, nbnd=16, per_atom=1, prec="fp64"),
        # 1000 coefficients continued to 20000 (bi-constant) on 4001 frequencies
        _spectrum_case("spectrum_osc"),
    ]


def draw(rng):
    """One more case: a cell on one of the grids it is run on, with a cut-off that the grid holds
    the products of, an uneven k-mesh, and the options in any combination; no more work than the
    largest listed one (an FP64 flop counted as four)."""
    while True:
        c = _draw(rng)
        if work(c)["flops"] * (4 if c.get("prec") == "fp64" else 1) <= 3.0e11:
            return c


def _draw(rng):
    if rng.random() < 0.15:
        m = round(math.exp(rng.uniform(math.log(40), math.log(3000))))
        return _spectrum_case(m=m, m_total=round(math.exp(rng.uniform(math.log(m), math.log(20000)))),
                              n_omega=round(math.exp(rng.uniform(math.log(50), math.log(8000)))),
                              extrap=rng.choice(["constant", "osc"]))
    cell = rng.choice(["fcc", "fcc", "fcc", "cubic", "super"])
    nfft, e0 = rng.choice({"fcc": [(12, 4.4), (16, 7.9), (18, 10.0), (24, 17.8), (32, 27.0), (36, 40.0)],
                           "cubic": [(24, 11.0), (32, 20.0), (36, 25.0)], "super": [(36, 17.0), (48, 30.0)]}[cell])
    kmax = {"fcc": 8, "cubic": 4, "super": 3}[cell] if nfft <= 32 else 3
    prec = rng.choice(["fp32", "fp32", "fp64"])
    k = [1 + math.floor(math.exp(rng.uniform(0, math.log(kmax)))) for _ in range(3)]
    k = [min(x, kmax) for x in k]
    metal = cell == "fcc" and nfft in (16, 18) and rng.random() < 0.25
    nbnd = 6 if metal else {"fcc": rng.choice([2, 3, 4, 5, 8]), "cubic": rng.choice([8, 13, 16]), "super": rng.choice([24, 32])}[cell]
    kind = "apply" if k[0] * k[1] * k[2] <= 64 and rng.random() < 0.2 else "chain"
    return _case(kind=kind, cell=cell, ecut=round(e0 * rng.uniform(0.7, 1.0), 4), nfft=nfft, k1=k[0], k2=k[1], k3=k[2], nbnd=nbnd,
                 per_atom=0 if metal else rng.choice([0, 1, 4]), prec=prec, flavour=rng.choice(["ph", "ph", "nh"]),
                 approx=rng.choice(["tddft", "tddft", "rpa", "ipa"]), q=round(rng.uniform(0.05, 0.6), 4),
                 steps=rng.choice([4, 6, 8]), stream=rng.random() < 0.6, wedge=cell == "fcc" and not metal and rng.random() < 0.2,
                 metal=metal)


# ---- the crystal: everything that does not depend on the seed ------------------------------
def _lattice(cell):
    if cell == "cubic":
        lat = A * np.eye(3)
        f = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
        return lat, np.concatenate([f, f + 0.25]) @ lat
    p = 0.5 * A * np.array([[-1., 0., 1.], [0., 1., 1.], [-1., 1., 0.]])
    tau = np.array([[0., 0., 0.], [A / 4] * 3])
    if cell == "fcc":
        return p, tau
    sh = [i * p[0] + j * p[1] + k * p[2] for i in range(2) for j in range(2) for k in range(2)]
    return 2 * p, np.array([t + s for s in sh for t in tau])


def _qvec(case):
    d = np.array([1., 0., 0.]) if case["cell"] != "super" else np.array([1., 1., 0.]) / math.sqrt(2)
    return case["q"] * (2 * np.pi / A) * d


def _group(lat):
    """Cartesian operations of C2v about x and their matrices on the FFT grid of an FCC cell."""
    ops = [np.eye(3), np.diag([1., -1., -1.]), np.array([[1., 0, 0], [0, 0, 1], [0, 1, 0]]),
           np.array([[1., 0, 0], [0, 0, -1], [0, -1, 0]])]
    inv = np.linalg.inv(lat.T)
    return ops, np.array([np.round(inv @ r @ lat.T) for r in ops]).astype(np.int32)


@lru_cache(maxsize=4)
def _crystal(cell, ecut, nfft, k1, k2, k3, q, wedge):
    lat, tau = _lattice(cell)
    b = 2 * np.pi * np.linalg.inv(lat).T
    n = np.array([k1, k2, k3])
    kf = np.stack(np.meshgrid(*[np.arange(x) / x for x in n], indexing="ij"), -1).reshape(-1, 3)
    weight = sym = None
    if wedge:       # stars of the mesh under the small group of Q, where the mesh has it
        ops, sym = _group(lat)
        keep = [i for i, r in enumerate(ops)
                if np.allclose(g := ((kf @ b) @ r.T @ np.linalg.inv(b)) * n, np.round(g), atol=1e-6)]
        ops, sym = [ops[i] for i in keep], np.ascontiguousarray(sym[keep])
        index = {tuple(x): i for i, x in enumerate(np.round(kf * n).astype(int))}
        star = [frozenset(index[tuple(np.round(((r @ (f @ b)) @ np.linalg.inv(b)) * n).astype(int) % n)] for r in ops) for f in kf]
        first = {s: i for i, s in reversed(list(enumerate(star)))}
        kf, weight = kf[sorted(first.values())], np.array([float(len(star[i])) for i in sorted(first.values())])
    kc = kf @ b
    qc = _qvec(dict(cell=cell, q=q))
    out = dict(lat=lat, tau=tau, b=b, kc=kc, qc=qc, omega=abs(np.linalg.det(lat)), weight=weight, sym=sym)
    for key, pts in (("k", kc), ("kq", kc + qc)):
        kmax = math.sqrt(ecut) + np.linalg.norm(pts, axis=1).max()
        mm = [int(kmax * np.linalg.norm(lat[i]) / (2 * np.pi)) + 1 for i in range(3)]
        m = np.stack(np.meshgrid(*[np.arange(-x, x + 1) for x in mm], indexing="ij"), -1).reshape(-1, 3)
        g = m @ b
        out["mil_" + key] = [np.ascontiguousarray(m[((p + g) ** 2).sum(1) <= ecut], dtype=np.int32) for p in pts]
    return out


class _Sphere:
    """Padded tables of one family of plane-wave spheres on the device."""

    def __init__(self, mil, pts, b, nfft):
        npw = [len(m) for m in mil]
        pad = max(npw)
        m = np.zeros((len(mil), pad, 3), dtype=np.int64)
        ok = np.zeros((len(mil), pad), dtype=bool)
        for i, x in enumerate(mil):
            m[i, :len(x)], ok[i, :len(x)] = x, True
        self.npw, self.pad = npw, pad
        self.ok = torch.from_numpy(ok).cuda()
        self.g = torch.from_numpy(m @ b + pts[:, None, :]).cuda()
        w = m % nfft
        self.flat = torch.from_numpy(np.where(ok, (w[..., 0] * nfft + w[..., 1]) * nfft + w[..., 2], nfft ** 3)).cuda()

    def packed(self, rows):
        """(nks, r, pad) -> the packed 1-D layout of the descriptor."""
        return rows[self.ok[:, None, :].expand(rows.shape)].contiguous()


def _orthonormal(u):
    """Rows of every k orthonormalised (Cholesky of the overlap, twice for rounding)."""
    for _ in range(2):
        s = u @ u.mH
        u = torch.linalg.solve_triangular(torch.linalg.cholesky(s), u, upper=False)
    return u


def _ground_state(case, seed):
    """The descriptor's arrays of one seeded model ground state, on the device."""
    c = _crystal(*[case[x] for x in ("cell", "ecut", "nfft", "k1", "k2", "k3", "q", "wedge")])
    rng = np.random.default_rng(seed)
    n, nb, nks = case["nfft"], case["nbnd"], len(c["kc"])
    om, lat, b = c["omega"], c["lat"], c["b"]
    sk = _Sphere(c["mil_k"], c["kc"], b, n)
    sq = _Sphere(c["mil_kq"], c["kc"] + c["qc"], b, n)
    tau = c["tau"] + rng.normal(0.0, 0.05, c["tau"].shape)
    nel = 8 if case["metal"] else 2 * nb
    # bond centres: a low-discrepancy set in the cell plus noise; width from their spacing
    phi = 1.2207440846057596
    cen = ((0.5 + np.arange(1, nb + 1)[:, None] * phi ** -np.arange(1., 4.)) % 1.0) @ lat + rng.normal(0.0, 0.1, (nb, 3))
    wid = 0.35 * (om / nb) ** (1 / 3)
    f = np.fft.fftfreq(n, 1.0 / n)
    g = torch.from_numpy(np.stack(np.meshgrid(f, f, f, indexing="ij"), -1) @ b).cuda()
    g2 = (g * g).sum(-1)
    box = (g2 > 0) & (g2 <= 4.0 * case["ecut"])
    phase = lambda pos: sum(torch.exp(-1j * (g @ torch.from_numpy(p).cuda())) for p in pos)
    shape = phase(cen) * torch.exp(-g2 * wid ** 2 / 4) / (om * nb)
    to_r = lambda x: torch.fft.ifftn(x, norm="forward").real
    rho = torch.clamp(to_r(nel * torch.where(box, shape, torch.zeros_like(shape))) + nel / om, min=2e-3)
    vg = 4 * np.pi / g2.clamp(min=1e-9) * (nel * shape - nel / len(tau) / om * phase(tau) * torch.exp(-g2 / 4))
    if c["sym"] is not None:    # the density has the group's symmetry
        j = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1)
        rho = sum(rho[tuple(torch.from_numpy(((j @ s.T) % n)).cuda().unbind(-1))] for s in c["sym"]) / len(c["sym"])
    vloc = to_r(torch.where(box, vg, torch.zeros_like(vg))) - (3 / np.pi * rho) ** (1 / 3)
    # Kleinman-Bylander projectors: repulsive s, weak attractive p on every atom
    beta = dij = None
    if case["per_atom"]:
        r = []
        for t in tau:
            x = torch.exp(-0.16 * (sq.g ** 2).sum(-1)) * torch.exp(-1j * (sq.g @ torch.from_numpy(t).cuda())) * sq.ok / math.sqrt(om)
            r.append(0.80 * x)
            if case["per_atom"] == 4:
                r += [-0.26j * sq.g[..., i] * x for i in range(3)]
        beta = torch.stack(r, 1)
        dij = np.array(([21.0, -0.5, -0.5, -0.5] if case["per_atom"] == 4 else [20.0]) * len(tau))
    vbox = torch.fft.fftn(vloc, norm="forward")

    def hamiltonian(mil, gv):
        d = torch.from_numpy((mil[:, None, :] - mil[None, :, :]) % n).cuda().long()
        return vbox[d[..., 0], d[..., 1], d[..., 2]] + torch.diag(0.5 * (gv ** 2).sum(-1))

    extra = {}
    if case["metal"]:            # eigenstates; the Fermi level below the bands left out
        lev = []
        for s, mil in ((sk, c["mil_k"]), (sq, c["mil_kq"])):
            h = torch.zeros(nks, s.pad, s.pad, dtype=torch.complex128, device="cuda")
            for i, x in enumerate(mil):
                h[i, :len(x), :len(x)] = hamiltonian(x, s.g[i, :len(x)])
                h[i, range(len(x), s.pad), range(len(x), s.pad)] = 1e3
            e, v = torch.linalg.eigh(h)
            lev.append((e, v.mT[:, :nb].contiguous()))
        (ek, uk), (eq, uq) = lev
        sig = 0.02
        mu = float(min(ek[:, nb].min(), eq[:, nb].min())) - 8 * sig
        occ = lambda e: (lambda f: torch.where(f < 1e-12, 0.0, torch.where(f > 1 - 1e-12, 1.0, f)))(0.5 * torch.erfc((e[:, :nb] - mu) / sig))
        extra = dict(occ_k=occ(ek).cpu().numpy(), occ_kq=occ(eq).cpu().numpy(), eps_kq=eq[:, :nb].cpu().numpy().copy())
        eps = ek[:, :nb].cpu().numpy().copy()
        z = torch.zeros(nks, nb, n ** 3 + 1, dtype=torch.complex128, device="cuda")
        z.scatter_(2, sk.flat[:, None, :].expand(uk.shape), uk)
        psi = torch.fft.ifftn(z[..., :-1].reshape(nks, nb, n, n, n), dim=(2, 3, 4), norm="forward")
        rho = (2 / om / nks) * (occ(ek)[..., None, None, None] * psi.abs() ** 2).sum((0, 1))
    else:
        amp = torch.from_numpy(rng.normal(0.0, 0.15, (nb, 4))).cuda()

        def bonds(s):
            g2 = (s.g ** 2).sum(-1)
            poly = torch.stack([torch.ones_like(g2), *(1j * wid * s.g).unbind(-1)], -1).to(torch.complex128)
            poly = torch.einsum("kgc,bc->kbg", poly, (amp + torch.tensor([1., 0, 0, 0], device="cuda")).to(torch.complex128))
            ph = torch.exp(-1j * torch.einsum("kgx,bx->kbg", s.g, torch.from_numpy(cen).cuda()))
            return _orthonormal(poly * ph * torch.exp(-0.5 * wid ** 2 * g2)[:, None, :] * s.ok[:, None, :])

        uk, uq = bonds(sk), bonds(sq)
        low = np.stack(np.meshgrid(*[np.arange(-8, 9)] * 3, indexing="ij"), -1).reshape(-1, 3)
        gl = low @ b
        low = low[np.argsort((gl ** 2).sum(1), kind="stable")[:300]]
        e0 = float(torch.linalg.eigvalsh(hamiltonian(low, torch.from_numpy(low @ b).cuda()))[0])
        eps = e0 - 0.3 - 0.1 * rng.random((1, nb)) - 0.05 * rng.random((nks, nb))
    return c, sk, sq, dict(lattice=lat, nfft=n, kcart=c["kc"], miller_k=c["mil_k"], miller_kq=c["mil_kq"], u_k=sk.packed(uk),
                           u_kq=sq.packed(uq), eps_k=np.ascontiguousarray(eps), vloc_r=vloc.contiguous(), rho_r=rho.contiguous(),
                           beta_kq=None if beta is None else sq.packed(beta), dij=dij, q_cart=c["qc"], approx=case["approx"],
                           flavour=case["flavour"], precision=case["prec"], kweight=c["weight"], sym=c["sym"], **extra), (uk, uq, beta)


def _coefficients(case, seed):
    """Coefficients of a finished chain: off-diagonals about half the cut-off energy with an
    even-odd splitting (the gap), z decaying."""
    rng = np.random.default_rng(seed)
    i = np.arange(case["m"])
    beta = 6.0 + 0.4 * (-1.0) ** i + rng.normal(0, 0.05, i.size)
    beta[0] = 0.3 + 0.2 * rng.random()
    z = np.where(i % 2, 0.3 * np.exp(-i / 150.0), 0.0) * np.exp(1j * rng.normal(0, 0.02, i.size)) * rng.choice([-1, 1], i.size)
    q = 0.1 * (2 * np.pi / A) * np.array([1., 0., 0.])
    return beta, beta.astype(np.complex128), z, 270.0, q, np.linspace(0.0, 40.0, case["n_omega"]), 0.1


def _batch(case, sq, nks, seed):
    rng = np.random.default_rng(seed + 1)
    n = case["nbnd"] * sum(sq.npw)
    return (rng.normal(size=n) + 1j * rng.normal(size=n)) / math.sqrt(max(sq.npw))


def prepare(case, seed):
    if case["kind"] == "spectrum":
        return dict(case=case, args=_coefficients(case, seed))
    c, sk, sq, system, _ = _ground_state(case, seed)
    s = dict(case=case, system=dict(system, max_steps=MAX_STEPS if case["kind"] == "chain" else 1),
             stream=torch.cuda.Stream() if case["stream"] else None)
    if case["kind"] == "apply":
        s["x"] = _batch(case, sq, len(c["kc"]), seed)
    torch.cuda.synchronize()
    s["chain"] = _open(s)
    return s


def _open(s):
    return ll.Chain(stream=s["stream"].cuda_stream if s["stream"] else None, **s["system"])


def run(state):
    case = state["case"]
    if case["kind"] == "spectrum":
        return ll.spectrum(*state["args"], extrapolation=case["extrap"], m_total=case["m_total"])
    if case["kind"] == "apply":
        out = state["chain"].apply(state["x"], case["approx"] != "ipa")
        return [x.astype(np.complex64) for x in out] if case["prec"] == "fp32" else out
    if state["chain"].steps + case["steps"] > MAX_STEPS:
        state["chain"].close()
        state["chain"] = _open(state)
    beta, gamma, z = state["chain"].lanczos(case["steps"])
    if case["prec"] == "fp32":
        return beta.astype(np.float32), gamma.astype(np.complex64), z.astype(np.complex64)
    return beta, gamma, z


def work(case):
    """Bytes: vectors, occupied states and projectors read once and vectors written once per
    application (the step's three vectors), the ground state's u_k on the D + K ones.  Flops: the
    line transforms that the spheres' columns, rows and planes need on the declared grid, and the
    projections."""
    if case["kind"] == "spectrum":
        return dict(bytes=40.0 * case["m"] + 56.0 * case["n_omega"], flops=30.0 * max(case["m"], case["m_total"]) * case["n_omega"])
    c = _crystal(*[case[x] for x in ("cell", "ecut", "nfft", "k1", "k2", "k3", "q", "wedge")])
    n, nb, nk = case["nfft"], case["nbnd"], len(c["kc"])
    npw = sum(len(m) for m in c["mil_kq"])
    npk = sum(len(m) for m in c["mil_k"])
    proj = case["per_atom"] * len(c["tau"])
    line = 5.0 * n * math.log2(n)
    cols = sum(len(np.unique(m[:, :2], axis=0)) for m in c["mil_kq"][:: max(1, nk // 16)]) * nk / len(c["mil_kq"][:: max(1, nk // 16)])
    rows = sum(len(np.unique(m[:, 1])) for m in c["mil_kq"][:: max(1, nk // 16)]) * nk / len(c["mil_kq"][:: max(1, nk // 16)])
    half = nb * (cols * line + n * (rows + n * nk) * line)          # one way between spheres and grids
    cs = 16.0 if case["prec"] == "fp64" else 8.0
    vec = cs * nb * npw
    gemm = 8.0 * npw * nb * (2 * nb + 2 * proj)
    d_bytes, d_flops = cs * npw * (nb + proj) + 8.0 * n ** 3, 2 * half + gemm + 2.0 * nb * nk * n ** 3
    k_bytes, k_flops = cs * nb * npk + 8.0 * n ** 3, half + 14.0 * nb * nk * n ** 3
    has_k = case["approx"] != "ipa"
    if case["kind"] == "apply":
        return dict(bytes=d_bytes + has_k * k_bytes + 32.0 * nb * npw, flops=d_flops + has_k * k_flops)
    steps, nv = case["steps"], 2 if case["flavour"] == "nh" else 1
    per = nv * 6 * vec + d_bytes + (1.0 if nv == 2 else 0.5) * has_k * k_bytes
    fl = nv * d_flops + (1.0 if nv == 2 else 0.5) * has_k * k_flops + 8.0 * npw * nb * nb * nv
    return dict(bytes=steps * per, flops=steps * fl)


# ---- the same results from plain torch in 64 bits ------------------------------------------
class _Exact:
    def __init__(self, case, seed):
        self.case = case
        c, self.sk, self.sq, d, (uk, uq, beta) = _ground_state(case, seed)
        self.n, self.nb, self.nks = case["nfft"], case["nbnd"], len(c["kc"])
        w = np.ones(self.nks) if c["weight"] is None else np.sqrt(c["weight"] * self.nks / c["weight"].sum())
        occ = d.get("occ_k", np.ones((self.nks, self.nb)))
        self.uk = uk * torch.from_numpy(w[:, None] * np.sqrt(occ)).cuda()[..., None]
        self.uq, self.beta, self.omega = uq, beta, c["omega"]
        self.dij = None if beta is None else torch.from_numpy(d["dij"]).cuda()
        self.eps = torch.from_numpy(d["eps_k"]).cuda()
        self.kin = 0.5 * (self.sq.g ** 2).sum(-1)
        self.v = d["vloc_r"]
        f = np.fft.fftfreq(self.n, 1.0 / self.n)
        g = torch.from_numpy(np.stack(np.meshgrid(f, f, f, indexing="ij"), -1) @ c["b"] + c["qc"]).cuda()
        self.wh = 4 * np.pi / (g * g).sum(-1)
        self.fxc = self._fxc(d["rho_r"]) if case["approx"] == "tddft" else None
        self.sym = c["sym"]
        self.metal = None
        if case["metal"]:
            fv, fm = occ[:, None, :], d["occ_kq"][:, :, None]
            cw = np.where(fv > 0, np.maximum(1 - fm / np.where(fv > 0, fv, 1), 0), 0.0)
            cw[cw < 1e-6] = 0.0
            qh = np.where(cw > 0, 1 - np.sqrt(cw), 0.0)
            da = np.where(cw > 0, (1 - cw) * (d["eps_kq"][:, :, None] - d["eps_k"][:, None, :]), 0.0)
            self.metal = [torch.from_numpy(x).cuda() for x in (np.where(cw > 0, qh, 1.0), da, (cw == 0) * 1.0, qh, (cw > 0) * 1.0)]
        nb_bytes = 16.0 * self.nb * (self.n ** 3 + 1)
        self.step = max(1, int(2e9 // nb_bytes))

    @staticmethod
    def _fxc(rho):
        """d v_xc/dn of Slater exchange and Perdew-Zunger 1981 correlation."""
        rs = (3 / (4 * math.pi * rho)) ** (1 / 3)
        fx = -4 / 9 * 0.75 * (3 / math.pi) ** (1 / 3) * rho ** (-2 / 3)
        g, b1, b2 = -0.1423, 1.0529, 0.3334
        s = rs.sqrt()
        den, dd, d2 = 1 + b1 * s + b2 * rs, b1 / (2 * s) + b2, -b1 / (4 * s ** 3)
        hi1, hi2 = -g * dd / den ** 2, -g * (d2 * den - 2 * dd * dd) / den ** 3
        lo1, lo2 = 0.0311 / rs + 0.0020 * (rs.log() + 1) - 0.0116, -0.0311 / rs ** 2 + 0.0020 / rs
        e1, e2 = torch.where(rs >= 1, hi1, lo1), torch.where(rs >= 1, hi2, lo2)
        return fx + (2 / 3 * e1 - rs / 3 * e2) * (-rs / (3 * rho))

    def grid(self, x, s, k):
        z = torch.zeros(x.shape[0], self.nb, self.n ** 3 + 1, dtype=torch.complex128, device="cuda")
        z.scatter_(2, s.flat[k][:, None, :].expand(x.shape), x)
        return torch.fft.ifftn(z[..., :-1].reshape(-1, self.nb, self.n, self.n, self.n), dim=(2, 3, 4), norm="forward")

    def gather(self, r, k):
        z = torch.fft.fftn(r, dim=(2, 3, 4), norm="forward").reshape(r.shape[0], self.nb, -1)
        idx = self.sq.flat[k].clamp(max=self.n ** 3 - 1)[:, None, :].expand(-1, self.nb, -1)
        return torch.gather(z, 2, idx) * self.sq.ok[k][:, None, :]

    def coef(self, u, x):
        return u.conj() @ x.mT        # [k][m][v]

    def project(self, x, weight=None):
        s = self.coef(self.uq, x)
        return x - (s if weight is None else s * weight).mT @ self.uq

    def op(self, z, upper):
        if self.metal:
            sp, da, _, qh, kept = self.metal
            zm = self.coef(self.uq, z)
            x = z - (qh * zm).mT @ self.uq
        else:
            x = z
        t = x * (self.kin[:, None, :] - self.eps[..., None])
        dens = torch.zeros(self.n, self.n, self.n, dtype=torch.complex128, device="cuda")
        parts = [slice(i, min(i + self.step, self.nks)) for i in range(0, self.nks, self.step)]
        for k in parts:
            r = self.grid(x[k], self.sq, k)
            t[k] += self.gather(r * self.v, k)
            if upper:
                dens += (self.grid(self.uk[k], self.sk, k).conj() * r).sum((0, 1))
        if upper:
            dens *= 4 / (self.omega * self.nks)
            if self.sym is not None:
                j = np.stack(np.meshgrid(*[np.arange(self.n)] * 3, indexing="ij"), -1)
                dens = sum(dens[tuple(torch.from_numpy((j @ s.T) % self.n).cuda().unbind(-1))] for s in self.sym) / len(self.sym)
            vp = torch.fft.ifftn(torch.fft.fftn(dens) * self.wh)
            if self.fxc is not None:
                vp = vp + self.fxc * dens
            for k in parts:
                t[k] += self.gather(self.grid(self.uk[k], self.sk, k) * vp, k)
        if self.beta is not None:
            t += (self.coef(self.beta, x) * self.dij[:, None]).mT @ self.beta
        if self.metal:
            return t - (sp * self.coef(self.uq, t) - da * kept * zm).mT @ self.uq
        return self.project(t)

    def start(self):
        y = torch.zeros(self.nks, self.nb, self.sq.pad, dtype=torch.complex128, device="cuda")
        for k in range(self.nks):
            z = torch.zeros(self.nb, self.n ** 3 + 1, dtype=torch.complex128, device="cuda")
            z[:, self.sk.flat[k]] = self.uk[k]
            z[:, -1] = 0
            y[k] = z[:, self.sq.flat[k]]
        if self.metal:
            return self.project(self.project(y, self.metal[2]), self.metal[3])
        return self.project(y)

    def inner(self, a, b):
        return complex(torch.vdot(a.reshape(-1), b.reshape(-1))) / self.nks

    def keep(self, x):
        return self.project(x, self.metal[2] if self.metal else None)

    def chain(self, steps):
        k_on = self.case["approx"] != "ipa"
        y = self.start()
        beta, gamma, z = np.zeros(steps), np.zeros(steps, complex), np.zeros(steps, complex)
        if self.case["flavour"] == "ph":
            r, prev = y.clone(), torch.zeros_like(y)
            x = self.op(r, False)
            for j in range(1, steps + 1):
                b = math.sqrt(self.inner(r, x).real)
                beta[j - 1] = gamma[j - 1] = b
                if j % 2 == 0:
                    z[j - 1] = self.inner(y, r) / b
                if j == steps:
                    break
                nxt = self.keep(x / b - prev * b)
                prev, r = r / b, nxt
                x = self.op(r, j % 2 == 1 and k_on)
            return beta, gamma, z
        b = math.sqrt(self.inner(y, y).real)
        v, w = y / b, y / b
        vp, wp, g = torch.zeros_like(y), torch.zeros_like(y), complex(b)
        for j in range(1, steps + 1):
            beta[j - 1], gamma[j - 1] = b, g
            up = j % 2 == 0
            if up:
                z[j - 1] = self.inner(y, v)
            if j == steps:
                break
            vh = self.keep(self.op(v, up and k_on) - g * vp)
            wh = self.keep(self.op(w, not up and k_on) - b * wp)
            s = self.inner(wh, vh)
            b = math.sqrt(abs(s))
            g = s / b
            vp, wp, v, w = v, w, vh / b, wh / np.conj(g)
        return beta, gamma, z


def _exact_spectrum(case, seed):
    beta, gamma, z, om, q, w, eta = _coefficients(case, seed)
    m, tot = case["m"], max(case["m"], case["m_total"])
    b, g, zz = np.zeros(tot), np.zeros(tot, complex), np.zeros(tot, complex)
    b[:m], g[:m], zz[:m] = beta, gamma, z
    h, i = max(1, m // 2), np.arange(m, tot)
    for p in (0, 1):
        pick = slice(h, m) if case["extrap"] == "constant" else np.arange(h + (h + p) % 2, m, 2)
        b[i[i % 2 == p]], g[i[i % 2 == p]] = beta[pick].mean(), gamma[pick].mean()
    wc = (w + 1j * eta) / HA_EV
    d, r = wc.copy(), np.full(wc.shape, zz[tot - 1])
    for j in range(tot - 2, -1, -1):
        d, r = wc - b[j + 1] * g[j + 1] / d, zz[j] + b[j + 1] * r / d
    chi = 4 / om * b[0] * r / d
    ei = 1 + 4 * np.pi / (q @ q) * chi
    return chi, ei, 1 / ei


def exact(case, seed):
    if case["kind"] == "spectrum":
        return _exact_spectrum(case, seed)
    e = _Exact(case, seed)
    if case["kind"] == "chain":
        return e.chain(case["steps"])
    x = torch.zeros(e.nks, e.nb, e.sq.pad, dtype=torch.complex128, device="cuda")
    x[e.sq.ok[:, None, :].expand(x.shape)] = torch.from_numpy(_batch(case, e.sq, e.nks, seed)).cuda()
    out = e.op(x, case["approx"] != "ipa").cpu().numpy()
    return [np.ascontiguousarray(out[k, :, :n]) for k, n in enumerate(e.sq.npw)]
