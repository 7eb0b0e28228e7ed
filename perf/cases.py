"""The calls by which the TC operator is measured, each through its public entry point.

A case is a dict of plain values: the call, the cell and its sizes.  ``prepare`` makes what a user's
program holds before the call (seeded orbitals on the device, the library context), ``run`` makes one
call, ``exact`` gives the same result in 64 bits from plain torch.

FP32 contexts compute in FP32 and hand their results over in the FP64 layout of the interface; a
program that asks for FP32 keeps them in 32 bits, so ``run`` returns those outputs as complex64 /
float32 and the FP64 contexts' as they come.
"""
import math
import random

import numpy as np
import torch

from paper_2302_07420_gb300 import synth
from paper_2302_07420_gb300.operator import BandContext, BatchContext, Context

BOXES = (9, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 48)


def listed():
    return [
        # the smallest call in earnest: the closed-shell 14-electron gas at Gamma, FP64 (launches and latency)
        dict(name="heg14_fp64", call="apply", cell="heg", n=16, k1=1, k2=1, k3=1, bands=7, occ=7, fp="fp64"),
        # one SCF update of the silicon-like cell on a coarse mesh, as in a first convergence test
        dict(name="si_k222_fp32", call="apply", cell="si", n=24, k1=2, k2=2, k3=2, bands=4, occ=4, fp="fp32"),
        # the production mesh of the silicon-like cell, FP32: the operator of every SCF iteration
        dict(name="si_k444_fp32", call="apply", cell="si", n=24, k1=4, k2=4, k3=4, bands=4, occ=4, fp="fp32"),
        # an odd mesh in FP64, the precision of reference runs and of the default context
        dict(name="si_k333_fp64", call="apply", cell="si", n=24, k1=3, k2=3, k3=3, bands=4, occ=4, fp="fp64"),
        # the production mesh with crystal symmetry and time reversal (8 of 64 k-points computed)
        dict(name="si_k444_sym_fp32", call="symmetric", cell="si", n=24, k1=4, k2=4, k3=4, bands=4, occ=4, fp="fp32"),
        # the large box: 114 electrons at Gamma, 57 bands on 48^3
        dict(name="heg114_fp32", call="apply", cell="heg", n=48, k1=1, k2=1, k3=1, bands=57, occ=57, fp="fp32"),
        # many independent cells of uneven size in one launch (a sweep over densities and boxes)
        dict(name="heg_cells_fp32", call="batch", cells=8, pick=0, fp="fp32"),
        # two points of a band structure off the SCF mesh
        dict(name="si_k333_band_fp32", call="band", cell="si", n=24, k1=3, k2=3, k3=3, bands=4, occ=4, fp="fp32",
             points=2),
        # the backward pass: orbital and Jastrow-parameter gradients of the energy (Jastrow optimisation)
        dict(name="si_k222_grad_fp64", call="grad", cell="si", n=24, k1=2, k2=2, k3=2, bands=4, occ=4, fp="fp64"),
        # one block-Davidson step, the eigensolver of the SCF loop, with empty bands
        dict(name="si_k122_davidson_fp64", call="davidson", cell="si", n=24, k1=1, k2=2, k3=2, bands=5, occ=4,
             fp="fp64"),
        # a triclinic cell on an odd box: ragged spheres, smeared occupations, empty bands
        dict(name="tri27_k123_fp32", call="apply", cell="tri", n=27, k1=1, k2=2, k3=3, bands=7, occ=5, fp="fp32"),
        # the energy alone on a small odd box (a total-energy scan)
        dict(name="tri15_energy_fp64", call="energy", cell="tri", n=15, k1=2, k2=1, k3=2, bands=3, occ=3, fp="fp64"),
    ]


def _cost(c):
    """Pair convolutions times box points, weighted by what a box size and a precision cost relative to 24^3 FP32."""
    if c["call"] == "batch":
        return sum(_cost(x) for x in _cells(c))
    nk = c["k1"] * c["k2"] * c["k3"]
    pairs = nk * c["occ"] * nk * c["bands"]
    if c["call"] == "band":
        pairs = nk * c["occ"] * (nk * c["occ"] + c["points"] * c["bands"])
    box = 7.0 if c["n"] == 48 else 3.0 if c["n"] >= 25 else 1.0
    call = {"grad": 6.0, "energy": 0.6, "davidson": 2.0}.get(c["call"], 1.0)
    return pairs * c["n"] ** 3 * box * call * (17.0 if c["fp"] == "fp64" else 1.0)


def draw(rng):
    while True:
        call = rng.choice(("apply",) * 5 + ("energy", "grad", "davidson", "band", "batch", "symmetric"))
        # (the Ritz vectors of a Davidson step amplify rounding by the inverse gaps: FP64 there)
        fp = "fp64" if call == "davidson" else rng.choice(("fp32", "fp32", "fp64"))
        if call == "batch":
            c = dict(call=call, cells=rng.randint(3, 10), pick=rng.randint(1, 10 ** 6), fp="fp32")
        else:
            cell = "si" if call == "symmetric" else rng.choice(("si", "heg", "tri"))
            m = rng.choice((2, 3)) if call == "symmetric" else 0
            n = rng.choice(BOXES if cell == "tri" else BOXES[3:-1] if cell == "heg" else (18, 20, 24, 25, 27))
            mesh = (m,) * 3 if m else tuple(rng.choice((1, 1, 2, 2, 3, 4)) for _ in range(3))
            occ = 4 if cell == "si" else int(round(math.exp(rng.uniform(math.log(2), math.log(33 if cell == "heg" else 9)))))
            bands = occ if cell == "heg" or m else occ + rng.choice((0, 0, 1, 3))
            c = dict(call=call, cell=cell, n=n, k1=mesh[0], k2=mesh[1], k3=mesh[2], bands=bands, occ=occ, fp=fp)
            if call == "band":
                c["points"] = rng.randint(1, 4)
            if n <= 12 and occ > 3:
                continue   # the spheres of the smallest boxes hold only a few bands
        if _cost(c) <= 2.5e9:
            return c


# ---------------------------------------------------------------------------
# cells, parameters and orbitals

def _cells(case):
    """The cells of a batch: gases of 14 to 66 electrons at r_s = 1 to 5 on boxes 16^3 to 32^3, 1 to 8 k-points."""
    rng = random.Random(case["pick"])
    boxes = [16, 18, 20, 24, 25, 27, 30, 32]
    got = []
    while len(got) < case["cells"]:
        n = boxes[len(got)] if case["pick"] == 0 else rng.choice(boxes)
        occ = rng.choice((7, 19, 27, 33))
        k = rng.choice(((1, 1, 1), (1, 1, 2), (1, 2, 2), (2, 2, 2)))
        c = dict(call="apply", cell="heg", n=n, k1=k[0], k2=k[1], k3=k[2], bands=occ, occ=occ, fp=case["fp"],
                 rs=round(rng.uniform(1.0, 5.0), 3))
        if _cost(c) <= 2.5e8:
            got.append(c)
    return got


def _params(c):
    n, occ = c["n"], c["occ"]
    if c["cell"] == "si":       # fcc, a = 10.26 bohr, 7.5 Ha at 24^3 and the same sphere-to-box ratio elsewhere
        lattice = 5.13 * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])
        ecut = 7.5 * (n / 24.0) ** 2
    elif c["cell"] == "heg":    # simple cubic; spheres |m| <= floor((n - 1) / 4), 12 at 48^3 (and r_s = 4 at 16^3, 2 at 48^3)
        rs = c.get("rs", 2.0 if n == 48 else 4.0)
        lattice = np.eye(3) * (2 * occ * 4.0 * np.pi / 3.0) ** (1.0 / 3.0) * rs
        r = 12 if n == 48 else 4 if n == 16 else (n - 1) // 4
        ecut = 0.5 * (r * 2.0 * np.pi / lattice[0, 0]) ** 2 * (1.0 + 1e-9)
    else:                       # triclinic, spheres of about a fifth of the box
        rng = np.random.default_rng(230207420 + 1000 * n + 10 * occ + c["k3"])
        lattice = 7.0 * (np.eye(3) + 0.1 * rng.standard_normal((3, 3)))
        ecut = 0.5 * (0.19 * n * 2.0 * np.pi / np.linalg.norm(lattice, axis=1).max()) ** 2
    omega = abs(np.linalg.det(lattice))
    a = math.sqrt(omega / (4.0 * math.pi * 2 * occ))          # Eqs. A_normalize and cusp
    return dict(lattice=lattice, kmesh=(c["k1"], c["k2"], c["k3"]), ecut=ecut, fft=(n,) * 3, nbands=c["bands"],
                nocc=occ, A=[a, a], C=[math.sqrt(2.0 * a), math.sqrt(a)])


def _mesh(kmesh):
    f = [np.where(np.arange(n) / n > 0.5, np.arange(n) / n - 1.0, np.arange(n) / n) for n in kmesh]
    return np.stack(np.meshgrid(*f, indexing="ij"), -1).reshape(-1, 3)


def _occupations(c, nk):
    occ = np.zeros((nk, c["bands"]))
    occ[:, : c["occ"]] = 1.0
    if c["cell"] == "tri" and c["occ"] > 1:       # smeared: the upper occupied bands are partly filled
        occ[:, c["occ"] - 1] = 0.4 + 0.1 * (np.arange(nk) % 4)
        occ[:, c["occ"] - 2] = 0.9
    return occ


def _orthonormal(p):
    for _ in range(2):
        p = torch.linalg.solve_triangular(torch.linalg.cholesky(p.conj().transpose(1, 2) @ p).conj().transpose(1, 2), p,
                                          upper=True, left=False)
    return p


def _orbitals(p, kfrac, npw, miller, seed):
    """Biorthonormal right and left orbitals [nk][bands][npw_max]: decaying random coefficients, chi 1 % off phi."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    B = 2.0 * np.pi * np.linalg.inv(p["lattice"]).T
    kg = torch.from_numpy((np.asarray(kfrac)[:, None, :] + miller) @ B).cuda()
    on = torch.arange(miller.shape[1], device="cuda")[None] < torch.from_numpy(np.asarray(npw, dtype=np.int64)).cuda()[:, None]
    damp = (torch.exp(-3.75 * (kg ** 2).sum(-1) / (2.0 * p["ecut"])) * on)[..., None]
    shape = (len(kfrac), miller.shape[1], p["nbands"])

    def noise():
        return damp * torch.randn(shape, generator=g, device="cuda", dtype=torch.complex128)

    phi, r = _orthonormal(noise()), noise()
    x = phi + 1e-2 * r / torch.linalg.vector_norm(r, dim=1, keepdim=True)
    chi = x @ torch.linalg.inv(phi.conj().transpose(1, 2) @ x)
    return phi.transpose(1, 2).contiguous(), chi.transpose(1, 2).contiguous()


def _band_points(n):
    return np.array([(0.13, 0.27, -0.31), (0.5, 0.0, 0.125), (-0.07, 0.41, 0.33), (0.21, -0.18, 0.06)])[:n]


def _symmetric_orbitals(p, ctx, kfrac, seed):
    """Eigenvectors of a symmetric one-body model at the irreducible points, unfolded over their stars."""
    rng = np.random.default_rng(seed)
    model = dict(v0=0.16 * rng.uniform(0.95, 1.05), w0=0.05 * rng.uniform(0.8, 1.2))
    npw, miller = ctx.layout()
    ctx.set_symmetry(synth.point_group(p["lattice"]), time_reversal=True)
    irr = sorted(set(int(k) for k in ctx.symmetry_info()[1][:, 0]))
    B = 2.0 * np.pi * np.linalg.inv(p["lattice"]).T
    f, x, _, gap = synth.model_orbitals(p["lattice"], kfrac[irr] @ B, [miller[k][: npw[k]] for k in irr], ctx.npw_max,
                                        p["nbands"], model=model)
    assert gap > 0.01
    phi = torch.zeros((ctx.nk, p["nbands"], ctx.npw_max), dtype=torch.complex128, device="cuda")
    chi = torch.zeros_like(phi)
    phi[irr], chi[irr] = torch.from_numpy(f).cuda(), torch.from_numpy(x).cuda()
    return ctx.symmetrize_orbitals(phi, chi)


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        cells = _cells(case)
        prm = [_params(c) for c in cells]
        ctx = BatchContext(prm, precision=case["fp"])
        orb = [_orbitals(p, _mesh(p["kmesh"]), l[2], l[3], seed * 97 + i) for i, (p, l) in enumerate(zip(prm, ctx.layouts))]
        return dict(case=case, ctx=ctx, phi=[o[0] for o in orb], chi=[o[1] for o in orb],
                    occ=[_occupations(c, l[0]) for c, l in zip(cells, ctx.layouts)])
    p = _params(case)
    if call == "band":
        kb = _band_points(case["points"])
        ctx = BandContext(kfrac_band=kb, precision=case["fp"], **p)
        phi, chi = _orbitals(p, np.concatenate([_mesh(p["kmesh"]), kb]), ctx.npw, ctx.miller, seed)
        m = ctx.nk_mesh
        return dict(case=case, ctx=ctx, phi=phi[:m].contiguous(), chi=chi[:m].contiguous(), occ=_occupations(case, m),
                    bphi=phi[m:].contiguous(), bchi=chi[m:].contiguous(), bocc=_occupations(case, case["points"]))
    ctx = Context(precision=case["fp"], **p)
    kfrac = _mesh(p["kmesh"])
    if call == "symmetric":
        phi, chi = _symmetric_orbitals(p, ctx, kfrac, seed)
    else:
        phi, chi = _orbitals(p, kfrac, ctx.npw, ctx.miller, seed)
    return dict(case=case, ctx=ctx, phi=phi, chi=chi, occ=_occupations(case, ctx.nk))


def run(s):
    case, ctx, call = s["case"], s["ctx"], s["case"]["call"]
    f32 = case["fp"] == "fp32"

    def kept(x):
        return x.to(torch.complex64) if f32 else x

    def number(x):
        return np.asarray(x, dtype=np.float32 if f32 else np.float64)

    if call == "energy":
        return {"energy": number(ctx.energy(s["phi"], s["chi"], s["occ"]))}
    if call == "grad":
        gp, gc, da, dc = ctx.energy_grad(s["phi"], s["chi"], s["occ"])
        return {"phi": kept(gp), "chi": kept(gc), "A": number(da), "C": number(dc)}
    if call == "davidson":
        phi, chi, eig, dim = ctx.davidson_step(s["phi"], s["chi"], s["occ"])
        return {"phi": kept(phi), "chi": kept(chi), "eig": eig.astype(np.complex64) if f32 else eig, "dim": dim}
    if call == "band":
        r, l = ctx.apply_band(s["phi"], s["chi"], s["occ"], s["bphi"], s["bchi"], s["bocc"])
        return {"right": kept(r), "left": kept(l)}
    if call == "batch":
        r, l = ctx.apply(s["phi"], s["chi"], s["occ"])
        return {"right": [kept(x) for x in r], "left": [kept(x) for x in l]}
    r, l = ctx.apply(s["phi"], s["chi"], s["occ"])
    return {"right": kept(r), "left": kept(l)}


def work(case):
    """Orbitals in and results out in the interface's FP64 layout and the kernel tables; the flops of the
    transforms that the method asks for (14 per pair chain, 4 per 3b4 pass, 14 per occupied pair)."""
    if case["call"] == "batch":
        w = [work(c) for c in _cells(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    p, n = _params(case), case["n"]
    k = p["kmesh"]
    nk, nb, no = k[0] * k[1] * k[2], case["bands"], case["occ"]
    npw = abs(np.linalg.det(p["lattice"])) * (2.0 * p["ecut"]) ** 1.5 / (6.0 * np.pi ** 2)
    z = 8 if case["fp"] == "fp32" else 16
    fft = 5.0 * n ** 3 * math.log2(n ** 3)
    out, pts = nk * nb, 0
    irr = nk
    if case["call"] == "band":
        pts, out = case["points"], case["points"] * nb
    if case["call"] == "symmetric":     # time reversal alone halves the mesh; the point group takes it further
        irr = {2: 3, 3: 4, 4: 8}[k[0]]
        out = irr * nb
    sides = {"energy": 1.0, "grad": 10.0, "davidson": 2.0}.get(case["call"], 2.0)
    flops = sides * nk * no * out * 18 * fft + (1.0 if sides == 2.0 else sides / 2) * nk * no * irr * no * 14 * fft
    deltas = np.prod([2 * m - 1 for m in k])
    return {"bytes": float(4 * (nk + pts) * nb * npw * 16 + deltas * 4 * n ** 3 * z / 2), "flops": float(flops)}


# ---------------------------------------------------------------------------
# the same results in 64 bits

def _spheres(p, kfrac):
    """Miller vectors of every sphere, lexicographic, and |k+G|."""
    B = 2.0 * np.pi * np.linalg.inv(p["lattice"]).T
    got = []
    for k in kfrac:
        b = [int(math.ceil((math.sqrt(2 * p["ecut"]) + np.linalg.norm(k @ B)) * np.linalg.norm(a) / (2 * np.pi))) + 1
             for a in np.asarray(p["lattice"])]
        m = np.stack(np.meshgrid(*[np.arange(-x, x + 1) for x in b], indexing="ij"), -1).reshape(-1, 3)
        kg = k @ B + m @ B
        got.append(m[0.5 * (kg * kg).sum(1) <= p["ecut"]])
    return got


def _aux(p, kcart):
    """(sum A_aux, sum p A_aux, alpha) over p = k + supercell reciprocal vectors, p = 0 left out."""
    S = np.asarray(p["lattice"]) * np.asarray(p["kmesh"])[:, None]
    near = np.stack(np.meshgrid(*[np.arange(-2, 3)] * 3, indexing="ij"), -1).reshape(-1, 3) @ S
    d = np.linalg.norm(near, axis=1)
    alpha = (d[d > 0].min() / 12.0) ** 2
    pmax = math.sqrt(-math.log(1e-20) / alpha) + np.linalg.norm(kcart)
    b = [int(math.ceil(pmax * np.linalg.norm(a) / (2 * np.pi))) + 1 for a in S]
    l = np.stack(np.meshgrid(*[np.arange(-x, x + 1) for x in b], indexing="ij"), -1).reshape(-1, 3)
    v = kcart - l @ (2.0 * np.pi * np.linalg.inv(S).T)
    q = (v * v).sum(1)
    v, q = v[q > 1e-20], q[q > 1e-20]
    w = np.exp(-alpha * q) / q
    return float(np.sum(np.sort(w))), (v * w[:, None]).sum(0), alpha


def _gradu2(g):
    """B(g) of Appendix B without cancellation (three ranges of g)."""
    s, m, l = g.clamp(max=1.0), g.clamp(1.0, 6.0), g.clamp(min=6.0)
    small = -0.25 * math.pi * s * s - (1 + 0.5 * s * s) * torch.atan(0.5 * s) + (1 + s * s) * torch.atan(s)
    mid = (1 + 0.5 * m * m) * torch.atan(2 / m) - (1 + m * m) * torch.atan(1 / m)
    large, t = torch.zeros_like(l), 1 / l ** 3
    for k in range(1, 60):
        large = large + (-1) ** k * ((2.0 ** (2 * k + 1) - 1) / (2 * k + 1) - (2.0 ** (2 * k + 2) - 1) / (2 * k + 3)) * t
        t = t / (l * l)
    return torch.where(g <= 1, small, torch.where(g <= 6, mid, large))


class _Exact:
    """One side of the operator (Sec. 2.6) in complex128; w2, w3 weigh the two- and three-body terms."""

    def __init__(self, case, p, phi, chi, occ, left, w2=1.0, w3=1.0, A=None, C=None, kb=None, bphi=None, bchi=None, bocc=None):
        self.p, self.left, self.s, self.w2, self.w3 = p, left, -1.0 if left else 1.0, w2, w3
        n = case["n"]
        kfrac = _mesh(p["kmesh"])
        self.nk, self.nb, self.no = len(kfrac), p["nbands"], p["nocc"]
        if kb is not None:
            kfrac = np.concatenate([kfrac, kb])
            phi, chi, occ = torch.cat([phi, bphi]), torch.cat([chi, bchi]), np.concatenate([occ, bocc])
        self.kfrac, self.B = kfrac, 2.0 * np.pi * np.linalg.inv(p["lattice"]).T
        self.kcart = kfrac @ self.B
        self.sph = _spheres(p, kfrac)
        self.om = abs(float(np.linalg.det(p["lattice"])))
        self.f = torch.from_numpy(np.asarray(occ)[:, : self.no].copy()).cuda()
        dev = dict(device="cuda", dtype=torch.float64)
        self.A = torch.tensor(p["A"], **dev) if A is None else A
        self.C = torch.tensor(p["C"], **dev) if C is None else C
        rep = np.where(np.arange(n) <= (n - 1) // 2, np.arange(n), np.arange(n) - n)
        self.G = torch.from_numpy(np.moveaxis(np.stack(np.meshgrid(rep, rep, rep, indexing="ij"), -1) @ self.B, -1, 0).copy()).cuda()
        self.n, self.N = n, n ** 3
        s0, _, alpha = _aux(p, np.zeros(3))
        self.gamma0 = self.om / (4 * math.sqrt(math.pi ** 3 * alpha)) - (-alpha + s0) / self.nk
        self.box = [torch.from_numpy(np.ravel_multi_index(tuple((m % n).T), (n,) * 3)).cuda() for m in self.sph]
        ket, bra = (chi, phi) if left else (phi, chi)
        self.ket = [self.real(ket[k][:, : len(m)], k) for k, m in enumerate(self.sph)]
        self.bra = [self.real(bra[k][:, : len(m)], k) for k, m in enumerate(self.sph)]
        self.gket = []
        for k, m in enumerate(self.sph):
            q = torch.from_numpy((self.kcart[k] + m @ self.B).T.copy()).cuda()
            self.gket.append(self.real(1j * q[None] * ket[k][:, None, : len(m)], k))
        self.tabs = {}

    def FT(self, x):
        return torch.fft.fftn(x, dim=(-3, -2, -1), norm="forward")

    def iFT(self, x):
        return torch.fft.ifftn(x, dim=(-3, -2, -1), norm="forward")

    def real(self, c, k):
        v = torch.zeros(c.shape[:-1] + (self.N,), dtype=torch.complex128, device="cuda")
        v[..., self.box[k]] = c
        return self.iFT(v.reshape(c.shape[:-1] + (self.n,) * 3))

    def u(self, q, s):
        c2 = 1 / self.C[s] ** 2
        return 4 * math.pi * self.A[s] * c2 / (q * (q + c2))

    def v2a(self, q, s):
        c2, g = 1 / self.C[s] ** 2, self.C[s] * torch.sqrt(q)
        lap = -4 * math.pi * self.A[s] * c2 / (q + c2)
        return 4 * math.pi / q + self.s * lap - 4 * math.pi * self.A[s] ** 2 / (self.C[s] * g) * _gradu2(g)

    def kern(self, k, q):
        """(p, V, u_pp, u_ap) / Omega at p = k - q + G."""
        d = self.kfrac[k] - self.kfrac[q]
        key = tuple(np.round(d * 5040).astype(int))
        if key not in self.tabs:
            pv = torch.from_numpy(d @ self.B).cuda()[:, None, None, None] + self.G
            q2 = (pv * pv).sum(0)
            zero = q2 < 1e-24
            q2 = torch.where(zero, 1.0, q2)
            v0 = -4 * math.pi * self.A[0] - 2 * math.pi * self.A[0] ** 2 / self.C[0] + 4 * math.pi * self.nk * self.gamma0
            self.tabs[key] = (pv, torch.where(zero, v0, self.v2a(q2, 0)) / self.om,
                              *[torch.where(zero, 0.0, self.u(q2, s)) / self.om for s in (0, 1)])
        return self.tabs[key]

    def corr(self, s):
        return (4 * math.pi * self.A[s]) ** 2 * self.gamma0 - (4 * math.pi * self.A[s] * self.C[s]) ** 2 / self.nk

    def conv(self, u, pv, F):
        """FT^{-1}[i p u F], a vector field."""
        return self.iFT(1j * pv * u * F[..., None, :, :, :])

    def div(self, u, pv, X):
        """-i u p . X for spectra X."""
        return -1j * u * (pv * X).sum(-4)

    def groups(self, count, other):
        g = max(1, int(3e8 // (other * 3 * self.N * 16)))
        return [slice(a, min(a + g, count)) for a in range(0, count, g)]

    def prepare(self):
        no, nk, S = self.no, self.nk, range(2)
        w = self.f / nk
        self.d = sum((w[k][:, None, None, None] * self.bra[k][:no].conj() * self.ket[k][:no]).sum(0) for k in range(nk))
        m = sum((w[k][:, None, None, None, None] * self.bra[k][:no, None].conj() * self.gket[k][:no]).sum(0) for k in range(nk))
        q2 = (self.G * self.G).sum(0)
        zero = q2 == 0
        q2 = torch.where(zero, 1.0, q2)
        self.us = [torch.where(zero, 0.0, self.u(q2, s)) for s in S]
        vh = torch.where(zero, 0.0, sum(self.v2a(q2, s) for s in S)) / self.om
        uh = (self.us[0] + self.us[1]) / self.om
        self.nt = self.FT(self.d)
        vH = self.iFT(vh * self.nt)
        self.h1 = self.conv(uh, self.G, self.nt)
        vb2 = self.iFT(self.div(uh, self.G, self.FT(m)))
        t3b1 = self.iFT(self.div(uh, self.G, self.FT(self.h1 * self.d)))
        h6, self.h3a, self.h3b = 0.0, [], []
        for k2 in range(nk):
            a, b, t = self.occupied(k2, w)
            h6 = h6 + t + self.corr_3a2(k2)
            self.h3a.append(a)
            self.h3b.append(b)
        h5 = sum((w[k][:, None, None, None, None] * self.h3b[k] * self.ket[k][:no, None]).sum(0) for k in range(nk))
        t3b2 = self.iFT(self.div(uh, self.G, self.FT(h5)))
        self.vloc = (self.w2 * (vH + self.s * vb2) +
                     self.w3 * (-0.5 * (self.h1 ** 2).sum(0) + 0.5 * h6 - t3b1 + t3b2))

    def occupied(self, k2, w):
        """h3 of both kinds for the occupied orbitals of k2 and their part of h6."""
        no = self.no
        ha, hb, h6 = 0.0, 0.0, 0.0
        for k1 in range(self.nk):
            pa, _, *ua = self.kern(k1, k2)
            pb, _, *ub = self.kern(k2, k1)
            for g in self.groups(no, no):
                f1 = w[k1][g]
                A = self.FT(self.bra[k2][:no, None].conj() * self.ket[k1][g][None])     # [q2, q1]
                Bt = self.FT(self.bra[k1][g][None].conj() * self.ket[k2][:no, None])     # [q2, q1]
                for s in range(2):
                    PA, PB = self.conv(ua[s], pa, A), self.conv(ub[s], pb, Bt)
                    if k2 < self.nk:
                        h6 = h6 + torch.einsum("a,b,abdxyz,abdxyz->xyz", w[k2].to(PA.dtype), f1.to(PA.dtype), PA, PB)
                    if s == 0:
                        c = f1[None, :, None, None, None, None]
                        ha = ha + (c * PB * self.ket[k1][g][None, :, None]).sum(1)
                        hb = hb + (c * PA * self.bra[k1][g][None, :, None].conj()).sum(1)
        return ha, hb, h6

    def corr_3a2(self, k):
        no, f = self.no, self.f[k].to(torch.complex128)
        F = self.FT(self.bra[k][:no, None].conj() * self.ket[k][:no][None])
        O = F[..., 0, 0, 0]
        F0 = torch.einsum("a,b,ab,ba->", f, f, O, O)
        Fab = torch.einsum("a,b,ba,abxyz->xyz", f, f, O, F) + torch.einsum("a,b,ab,baxyz->xyz", f, f, O, F)
        return sum(self.corr(s) * F0 + 4 * math.pi * self.A[s] / self.nk * self.iFT(self.us[s] * Fab)
                   for s in range(2)) / (self.nk * self.om ** 2)

    def pass_3b4(self, k, w):
        out = 0.0
        for kq in range(self.nk):
            pv, _, u, _ = self.kern(k, kq)
            for g in self.groups(self.no, w.shape[0]):
                Y = self.iFT(self.div(u, pv, self.FT(self.bra[kq][g][:, None, None].conj() * w[None])))
                out = out + ((self.f[kq][g] / self.nk)[:, None, None, None, None] * self.ket[kq][g][:, None] * Y).sum(0)
        return out

    def output(self, k):
        """Real-space output of every band at k, before the projection."""
        no, w2, w3, s2b = self.no, self.w2, self.w3, self.s
        ket, gket = self.ket[k], self.gket[k]
        Y = w3 * self.h1[None] * ket[:, None] - w2 * s2b * gket
        acc, w = 0.0, 0.0
        for kq in range(self.nk):
            pv, V, up, ua = self.kern(k, kq)
            for g in self.groups(no, ket.shape[0]):
                f = (self.f[kq][g] / self.nk)[:, None, None, None, None]
                bc, kq_ = self.bra[kq][g].conj(), self.ket[kq][g][:, None]
                F = self.FT(bc[:, None] * ket[None])
                b = self.conv(up, pv, F)
                Z = -(w2 * s2b * self.gket[kq][g] + w3 * self.h3a[kq][g])
                acc = acc + (f * (Z[:, None] * b).sum(2)).sum(0)
                w = w + (f[..., None] * kq_[:, :, None] * b).sum(0)
                X = bc[:, None, None] * Y[None] - w3 * ket[None, :, None] * self.h3b[kq][g][:, None] + w3 * self.d * b
                D = self.div(up, pv, self.FT(X)) - w2 * V * F
                D = D + w3 * self.div(ua, pv, self.FT(self.d * self.conv(ua, pv, F)))
                acc = acc + (f * kq_ * self.iFT(D)).sum(0)
        if k >= self.nk:
            acc, w = self.band_corr(k, acc, w)
        else:
            acc = acc + w3 * self.corr_3b6(k)
        acc = acc - w3 * self.pass_3b4(k, w)
        return acc + self.vloc * ket + w2 * s2b * (self.h1 * gket).sum(1) + w3 * (self.h1 * w).sum(1)

    def corr_3b6(self, k, W=None, gamma=None):
        no = self.no
        F = self.FT(self.bra[k][:no, None].conj() * self.ket[k][None])
        O = F[..., 0, 0, 0]
        neg = torch.roll(torch.flip(self.nt, (0, 1, 2)), (1, 1, 1), (0, 1, 2))
        out = 0.0
        for s in range(2):
            c, a = self.corr(s), 4 * math.pi * self.A[s] / self.nk
            us = self.us[s]
            if W is not None:
                c, a, us = (4 * math.pi * self.A[s]) ** 2 * gamma, -a, us * torch.einsum("dxyz,d->xyz", self.G, W)
            X = (us * F * neg).sum((-3, -2, -1))
            field = (O * c * self.nt[0, 0, 0] + a * X)[..., None, None, None] + a * O[..., None, None, None] * self.iFT(us * self.nt)
            out = out + (self.f[k][:, None, None, None, None] * self.ket[k][:no, None] * field).sum(0)
        return out / self.om ** 2

    def band_corr(self, k, acc, w):
        """Band forms of the divergence corrections (Eqs. divcorr_2ax_band to 3b6_div_band3); w includes its own."""
        no = self.no
        s1, Wn, alpha = _aux(self.p, self.kcart[k])
        gamma = self.om / (4 * math.sqrt(math.pi ** 3 * alpha)) - s1 / self.nk
        W = torch.from_numpy(Wn).cuda()
        Wc = W.to(torch.complex128)
        c = 4 * math.pi * float(self.A[0]) / (self.nk * self.om)
        f = self.f[k].to(torch.complex128)
        km, bm, ket = self.ket[k][:no], self.bra[k][:no].conj(), self.ket[k]
        fO = f[:, None] * (bm[:, None] * ket[None]).mean((-3, -2, -1))
        sc = lambda x: (x * 1.0).mean((-3, -2, -1))   # noqa: E731
        dotW = lambda x: torch.einsum("...dxyz,d->...xyz", x, Wc)   # noqa: E731
        mix = lambda a, x: torch.einsum("mj,mxyz->jxyz", a, x)   # noqa: E731
        acc = acc - 4 * math.pi * gamma / self.om * mix(fO, km)
        acc = acc + self.s * 1j * c * mix(fO, dotW(self.gket[k][:no]))
        acc = acc - self.s * 1j * c * mix(f[:, None] * sc(bm[:, None] * dotW(self.gket[k])[None]), km)
        hW = dotW(self.h1)
        acc = acc + 1j * c * mix(f[:, None] * sc(bm[:, None] * hW * ket[None]), km)
        ha, hb, _ = self.occupied(k, self.f / self.nk)
        Ob = (bm[:, None] * km[None]).mean((-3, -2, -1))
        ha = ha - 1j * c * torch.einsum("d,pm,pxyz->mdxyz", Wc, f[:, None] * Ob, km)
        hb = hb + 1j * c * torch.einsum("d,mp,pxyz->mdxyz", Wc, Ob * f[None], bm)
        acc = acc + 1j * c * mix(fO, dotW(ha))
        acc = acc - 1j * c * mix(f[:, None] * sc(ket[None] * dotW(hb)[:, None]), km)
        wc = -1j * c * Wc[None, :, None, None, None] * mix(fO, km)[:, None]
        w = w + wc       # enters 3a3 and 3b4
        acc = acc - 1j * c * mix(f[:, None] * sc(bm[:, None] * dotW(w)[None]), km)
        return acc + self.corr_3b6(k, W, gamma), w

    def project(self, k, width):
        v = self.FT(self.output(k)).reshape(self.nb, self.N)[:, self.box[k]]
        return torch.nn.functional.pad(v, (0, width - v.shape[1]))

    def apply(self, width, points=None):
        self.prepare()
        return torch.stack([self.project(k, width) for k in (range(self.nk) if points is None else points)])


def _kinetic(p, npw_max):
    kfrac = _mesh(p["kmesh"])
    B = 2.0 * np.pi * np.linalg.inv(p["lattice"]).T
    t = np.zeros((len(kfrac), npw_max))
    for k, m in enumerate(_spheres(p, kfrac)):
        q = (kfrac[k] + m) @ B
        t[k, : len(m)] = 0.5 * (q * q).sum(1)
    return torch.from_numpy(t).cuda()[:, None]


def _energy(case, p, s, **kw):
    g = _Exact(case, p, s["phi"], s["chi"], s["occ"], False, 0.5, 1.0 / 3.0, **kw).apply(s["phi"].shape[2])
    g = g + _kinetic(p, s["phi"].shape[2]) * s["phi"]
    occ = torch.from_numpy(s["occ"]).cuda()[..., None]
    return 2.0 / len(s["phi"]) * (occ * (s["chi"].conj() * g).real).sum()


def _davidson_eig(case, p, s):
    """Ritz values and subspace dimensions of one block-Davidson step."""
    phi, chi, occ, no, nb = s["phi"], s["chi"], s["occ"], case["occ"], case["bands"]
    t = _kinetic(p, phi.shape[2])

    def h(v):
        q = dict(p, nbands=no + nb)
        a, b = torch.cat([phi[:, :no], v], 1), torch.cat([chi[:, :no], v], 1)
        return t * v + _Exact(case, q, a, b, occ, False).apply(phi.shape[2])[:, no:]

    hv = h(phi)
    eps = (phi.conj() * hv).sum(-1, keepdim=True)
    x = t / (phi.abs() ** 2 * t).sum(-1, keepdim=True)
    a = 27 + 18 * x + 12 * x ** 2 + 8 * x ** 3
    w = a / (a + 16 * x ** 4) * (hv - eps * phi)
    dims, new = [], torch.zeros_like(phi)
    for k in range(len(phi)):
        basis = list(phi[k])
        for i in range(nb):
            r = w[k, i]
            for _ in range(2):
                for v in basis:
                    r = r - torch.vdot(v, r) * v
            if torch.linalg.vector_norm(r) >= 1e-8:
                new[k, len(basis) - nb] = r / torch.linalg.vector_norm(r)
                basis.append(new[k, len(basis) - nb])
        dims.append(len(basis))
    hw = h(new)
    eig = []
    for k, d in enumerate(dims):
        b, hb = torch.cat([phi[k], new[k, : d - nb]]), torch.cat([hv[k], hw[k, : d - nb]])
        lam = np.linalg.eigvals((b.conj() @ hb.T).cpu().numpy())
        eig.append(lam[np.argsort(lam.real, kind="stable")][:nb])
    return np.array(eig), np.array(dims, dtype=np.int32)


def exact(case, seed):
    s = prepare(case, seed)
    s["ctx"].close()
    call = case["call"]
    if call == "batch":
        both = [[], []]
        for c, phi, chi, occ in zip(_cells(case), s["phi"], s["chi"], s["occ"]):
            for side in (0, 1):
                both[side].append(_Exact(c, _params(c), phi, chi, occ, side == 1).apply(phi.shape[2]))
        return {"right": both[0], "left": both[1]}
    p, phi, chi, occ = _params(case), s["phi"], s["chi"], s["occ"]
    if call == "energy":
        return {"energy": np.float64(_energy(case, p, s))}
    if call == "davidson":     # the vectors' phases are free
        eig, dim = _davidson_eig(case, p, s)
        return {"phi": None, "chi": None, "eig": eig, "dim": dim}
    if call == "band":
        kb = _band_points(case["points"])
        nk = len(phi)
        r, l = [_Exact(case, p, phi, chi, occ, side, kb=kb, bphi=s["bphi"], bchi=s["bchi"], bocc=s["bocc"])
                .apply(phi.shape[2], range(nk, nk + len(kb))) for side in (False, True)]
        return {"right": r, "left": l}
    if _cost(dict(case, fp="fp32")) > 4e9:      # over about 20 s
        return None
    r, l = [_Exact(case, p, phi, chi, occ, side).apply(phi.shape[2]) for side in (False, True)]
    if call != "grad":
        return {"right": r, "left": l}
    t, f = _kinetic(p, phi.shape[2]), 2.0 / len(phi) * torch.from_numpy(occ).cuda()[..., None]
    A, C = [torch.tensor(p[x], device="cuda", dtype=torch.float64, requires_grad=True) for x in "AC"]
    if _cost(dict(case, fp="fp32")) > 6e8:      # the graph of the energy would not fit
        dA = dC = None
    else:
        _energy(case, p, s, A=A, C=C).backward()
        dA, dC = A.grad.cpu().numpy(), C.grad.cpu().numpy()
    return {"phi": f * (t * chi + l), "chi": f * (t * phi + r), "A": dA, "C": dC}
