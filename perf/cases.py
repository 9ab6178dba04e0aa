"""Workloads of the scattering-rate library, each through a public entry point of the package.

The crystals are seeded Morse solids: the two-atom diamond cell (a = 5.43 Å, m = 28.0855 amu,
D = 2 eV, α = 1.5/Å, r0 = 2.35 Å) or its 1x1xk supercell with masses in 10..120 amu, radial
derivatives of every bond perturbed by 1 %; Φ2 over the first neighbour shell, Φ3 and Φ4 over two.
A seed fixes the perturbations, the masses, the sampled q points and the Γ of the κ calls."""
import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2510_00518_gb300 as fc4

HBAR, EV, AMU, KB = 1.054571817e-34, 1.602176634e-19, 1.66053906660e-27, 1.380649e-23
EIG_TO_W2 = EV / (1e-20 * AMU) * 1e-24                      # eV/(Å² amu) -> (rad/ps)²
C3 = HBAR * math.pi / 4 * (EV / 1e-30 / AMU ** 1.5) ** 2 * 1e-60
C4 = HBAR ** 2 * math.pi / 8 * (EV / 1e-40 / AMU ** 2) ** 2 * 1e-72
A0, MORSE_D, MORSE_A, MORSE_R = 5.43, 2.0, 1.5, 2.35


def _case(kind, n1, n2, n3, precision="mixed", n_q=0, mask=31, adaptive=False, sigma=0.1, atoms=2, T=300.0,
          sampling=1.0, iters=0, name=None):
    """n_q = 0: the whole mesh; sigma: THz, or the scale factor of the adaptive width."""
    c = dict(kind=kind, n1=n1, n2=n2, n3=n3, precision=precision, n_q=n_q, mask=mask, adaptive=adaptive, sigma=sigma,
             atoms=atoms, T=T, sampling=sampling, iters=iters)
    return dict(c, name=name) if name else c


def listed():
    return [
        # κ of a converged Γ and its gradient: the smallest call, where launches and latency count
        _case("kappa", 16, 16, 16, "fp64", name="kappa_16cubed"),
        # one q point through the allocation-free entry point, as a latency-bound loop calls it
        _case("static", 6, 6, 6, n_q=1, name="static_1q_6cubed"),
        # a three-phonon calculation from force constants to κ, context set-up included
        _case("whole", 8, 8, 8, "fp64", mask=3, name="whole_3ph_8cubed"),
        # three-phonon rates alone, all modes of a production mesh
        _case("rates", 12, 12, 12, "fp64", mask=3, name="rates3_12cubed"),
        # three- and four-phonon rates of all modes, fixed width: the full calculation at mixed precision
        _case("rates", 8, 8, 8, name="rates_8cubed_mixed"),
        # sampled q points of a fine mesh, adaptive width: the form large meshes are run in
        _case("rates", 16, 16, 16, n_q=2, adaptive=True, sigma=1.0, name="rates_2q_16cubed_adaptive"),
        # the FP64 reference on sampled q points
        _case("rates", 8, 8, 8, "fp64", n_q=4, T=700.0, name="rates_4q_8cubed_fp64"),
        # FP16x3 contraction on the tensor cores, all modes
        _case("rates", 6, 6, 6, "fp16x3", name="rates_6cubed_fp16x3"),
        # eight atoms per cell (24 branches)
        _case("rates", 4, 4, 4, n_q=1, atoms=8, name="rates_1q_cell8_4cubed"),
        # four atoms per cell on a ragged mesh, adaptive width
        _case("rates", 5, 5, 4, n_q=3, atoms=4, adaptive=True, sigma=1.0, name="rates_3q_cell4_adaptive"),
        # κ and its gradient with respect to Φ3 and Φ4 through autograd
        _case("grad", 4, 4, 4, "fp64", name="grad_4cubed_fp64"),
        # iterative Boltzmann equation
        _case("bte", 4, 4, 4, iters=3, name="bte_4cubed_mixed"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mesh(rng, lo, hi):
    n = _log(rng, lo, hi)
    m = [max(lo, min(hi, round(n + rng.uniform(-0.7, 0.7)))) for _ in range(3)]
    return m if rng.random() < 0.6 else [m[0]] * 3


def _kept(case, na):
    """Rough share of the candidates of a channel pair (+-, then ++ and --) inside the window."""
    wide = 0.6 if case["adaptive"] else case["sigma"] / 0.1
    return 0.08 * wide, 0.002 * wide


def _modes(case):
    n = case["n1"] * case["n2"] * case["n3"]
    return n, 3 * case["atoms"], (case["n_q"] or n) * 3 * case["atoms"]


def _clusters(na):
    return 49 * na, 113 * na, 17 * na                        # Φ3, Φ4 clusters; fourth-order keys


def _flops(case):
    """Flops of one rates pass that keeps what the window keeps: window, cluster sums, V, weights."""
    n, nb, nm = _modes(case)
    nc3, nc4, keys = _clusters(case["atoms"])
    pm, sparse = _kept(case, case["atoms"])
    f = 0.0
    pairs = nm * n
    if case["mask"] & 3:
        kept = 2 * pairs * nb * nb * 0.02
        f += 2 * (2 * pairs * nb * nb) + min(kept, 2 * pairs) * keys * 72 + kept * (8 * nb + 30)
    for ch, share in ((2, sparse), (3, pm), (4, sparse)):
        if (case["mask"] >> ch) & 1:
            frac = 0.5 * case["sampling"]                    # partner-swap symmetry
            cand = pairs * n * nb ** 3 * frac
            entries = min(cand * share, pairs * n * nb * frac)
            items = min(cand * share, entries * nb)
            f += 2 * cand + pairs * (nc4 * 27 * 8 + nb * keys * 9 * nb * 8) + entries * keys * 72 + items * nb * nb * 8
            f += cand * share * (8 * nb + 30)
    return f


def _seconds(case):
    """Rough time of a pass, to keep drawn cases below the largest listed one."""
    f = _flops(case)
    rate = 1.5e11 if case["precision"] == "fp64" and case["mask"] & 28 else 3e12
    if case["precision"] not in ("fp64", "mixed"):
        rate = 2e12
    if case["atoms"] > 2:
        rate = min(rate, 4e11 if case["precision"] == "mixed" else 8e10)
    if case["adaptive"]:
        rate *= 0.7
    f *= {"grad": 12.0, "bte": max(1, case["iters"]) * 1.5 + 1.0}.get(case["kind"], 1.0)
    return f / rate


def draw(rng):
    while True:
        kind = rng.choice(["rates"] * 6 + ["rates3"] * 2 + ["kappa", "static", "whole", "grad", "bte"])
        T = round(rng.uniform(150.0, 900.0), 1)
        ad = rng.random() < 0.4
        sg = round(rng.uniform(0.7, 1.3), 2) if ad else round(_log(rng, 0.03, 0.15), 3)
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64", "fp64", "fp16x3", "tf32x3"])
        if kind == "kappa":
            c = _case("kappa", *_mesh(rng, 4, 20), "fp64", T=T)
        elif kind == "static":
            c = _case("static", *_mesh(rng, 3, 8), rng.choice(["mixed", "fp64"]), n_q=rng.choice([1, 1, 2, 3]), T=T,
                      sigma=round(_log(rng, 0.03, 0.15), 3))
        elif kind in ("whole", "rates3"):
            c = _case("whole" if kind == "whole" else "rates", *_mesh(rng, 4, 14), "fp64", mask=3, T=T, adaptive=ad, sigma=sg,
                      n_q=0 if kind == "whole" else rng.choice([0, 0, 1, 8, 29]), atoms=rng.choice([2, 2, 4]))
        elif kind == "rates":
            atoms = rng.choice([2, 2, 2, 2, 2, 4, 6, 8])
            c = _case("rates", *_mesh(rng, 3 if atoms > 2 else 4, 14 if atoms == 2 else 6), prec if atoms == 2 else "mixed",
                      n_q=rng.choice([0, 1, 2, 3, 7, 29]), adaptive=ad, sigma=sg, T=T, atoms=atoms,
                      sampling=rng.choice([1.0, 1.0, 1.0, 0.1]))
        elif kind == "grad":
            c = _case("grad", *_mesh(rng, 3, 5), rng.choice(["mixed", "fp64"]), adaptive=ad, sigma=sg, T=T)
        else:
            c = _case("bte", *_mesh(rng, 3, 5), rng.choice(["mixed", "fp64"]), iters=rng.choice([1, 3, 8]), T=T,
                      adaptive=ad, sigma=sg)
        n, _, nm = _modes(c)
        if c["n_q"] <= n and _seconds(c) < 0.3 and (c["kind"] != "static" or nm * n <= 65536):
            return c


# ------------------------------------------------------------------------------- inputs

def _crystal(atoms, rng):
    lat = 0.5 * A0 * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])
    k = atoms // 2
    base = np.array([[0.0, 0.0, 0.0], [0.25 * A0] * 3])
    pos = np.concatenate([base + m * lat[2] for m in range(k)])
    lat = np.stack([lat[0], lat[1], k * lat[2]])
    masses = np.full(2, 28.0855) if k == 1 else rng.uniform(10.0, 120.0, size=atoms)
    return SimpleNamespace(lattice=lat, positions=pos, masses=masses)


def _bonds(cr, cutoff):
    R = np.array(list(itertools.product(range(-3, 4), repeat=3)))
    out = []
    for i, j in itertools.product(range(len(cr.masses)), repeat=2):
        d = cr.positions[j] - cr.positions[i] + R @ cr.lattice
        r = np.linalg.norm(d, axis=1)
        out += [(i, j, tuple(int(x) for x in R[k]), d[k], r[k]) for k in np.nonzero((r > 1e-8) & (r < cutoff))[0]]
    return out


def _pair_tensor(order, d, r, p):
    """Cartesian derivatives of φ(|d|) from its radial derivatives p = (φ', φ'', φ''', φ'''')."""
    h1, h2 = p[0] / r, p[1] / r ** 2 - p[0] / r ** 3
    h3 = p[2] / r ** 3 - 3 * p[1] / r ** 4 + 3 * p[0] / r ** 5
    h4 = p[3] / r ** 4 - 6 * p[2] / r ** 5 + 15 * p[1] / r ** 6 - 15 * p[0] / r ** 7
    eye, dd = np.eye(3), np.multiply.outer(d, d)
    if order == 2:
        return h2 * dd + h1 * eye
    if order == 3:
        x = np.multiply.outer(eye, d)
        return h3 * np.multiply.outer(dd, d) + h2 * (x + x.transpose(0, 2, 1) + x.transpose(2, 0, 1))
    ed, ee = np.multiply.outer(eye, dd), np.multiply.outer(eye, eye)
    six = sum(ed.transpose(t) for t in ((0, 1, 2, 3), (0, 2, 1, 3), (0, 2, 3, 1), (2, 0, 1, 3), (2, 0, 3, 1), (2, 3, 0, 1)))
    three = ee + ee.transpose(0, 2, 1, 3) + ee.transpose(0, 2, 3, 1)
    return h4 * np.multiply.outer(dd, dd) + h3 * six + h2 * three


def _clusters_of(cr, order, cutoff, factors):
    acc = {}
    for i, j, R, d, r in _bonds(cr, cutoff):
        x = math.exp(-MORSE_A * (r - MORSE_R))
        p = 2 * MORSE_D * np.array([MORSE_A * (x - x * x), MORSE_A ** 2 * (2 * x * x - x), MORSE_A ** 3 * (x - 4 * x * x),
                                    MORSE_A ** 4 * (8 * x * x - x)])
        t = _pair_tensor(order, d, r, p * factors[min((i, j, R), (j, i, tuple(-v for v in R)))]).reshape(-1)
        for legs in itertools.product((0, 1), repeat=order - 1):
            key = ((i,) + tuple(j if g else i for g in legs), tuple(R if g else (0, 0, 0) for g in legs))
            acc[key] = acc.get(key, 0.0) + (-1.0) ** (order - sum(legs)) * t
    keys = sorted(acc)
    return SimpleNamespace(order=order, atoms=np.array([k[0] for k in keys], np.int32),
                           cells=np.array([k[1] for k in keys], np.int32), phi=np.array([acc[k] for k in keys]))


def _system(case, seed):
    """Crystal and its Φ2, Φ3, Φ4."""
    rng = np.random.default_rng([seed, 1])
    cr = _crystal(case["atoms"], rng)
    nn, nn2, nn3 = A0 * math.sqrt(3) / 4, A0 / math.sqrt(2), A0 * math.sqrt(11) / 4
    cut2, cut34 = 0.5 * (nn + nn2), 0.5 * (nn2 + nn3)
    classes = sorted({min((i, j, R), (j, i, tuple(-v for v in R))) for i, j, R, _, _ in _bonds(cr, cut34)})
    factors = {k: 1.0 + 0.01 * rng.uniform(-1.0, 1.0, size=4) for k in classes}
    return cr, _clusters_of(cr, 2, cut2, factors), _clusters_of(cr, 3, cut34, factors), _clusters_of(cr, 4, cut34, factors)


def _grid(mesh):
    i = np.arange(mesh[0] * mesh[1] * mesh[2])
    return np.stack([i % mesh[0], i // mesh[0] % mesh[1], i // (mesh[0] * mesh[1])], axis=1)


def _harmonic(cr, phi2, mesh):
    """ω [N, nb] rad/ps, v [N, nb, 3] Å/ps and e [N, component, branch] of the mesh."""
    frac = _grid(mesh) / np.asarray(mesh, float)
    nb = 3 * len(cr.masses)
    D = np.zeros((len(frac), nb, nb), complex)
    dD = np.zeros((3, len(frac), nb, nb), complex)
    for (a, b), cell, phi in zip(phi2.atoms, phi2.cells[:, 0], phi2.phi):
        f = np.exp(2j * np.pi * (frac @ cell)) / math.sqrt(cr.masses[a] * cr.masses[b])
        blk = f[:, None, None] * phi.reshape(3, 3)
        D[:, 3 * a:3 * a + 3, 3 * b:3 * b + 3] += blk
        R = cell @ cr.lattice
        for x in range(3):
            dD[x, :, 3 * a:3 * a + 3, 3 * b:3 * b + 3] += 1j * R[x] * blk
    lam, e = np.linalg.eigh(0.5 * (D + D.conj().transpose(0, 2, 1)))
    lam[0, :3] = 0.0
    w = np.sqrt(np.abs(lam) * EIG_TO_W2)
    dD = 0.5 * (dD + dD.conj().transpose(0, 1, 3, 2))
    v = np.einsum("qkj,xqkl,qlj->qjx", e.conj(), dD, e, optimize=True).real * EIG_TO_W2
    v = np.where(w[..., None] > 0, v / np.where(w > 0, 2 * w, 1.0)[..., None], 0.0)
    return w, v, e


def _subset(case, seed):
    n = case["n1"] * case["n2"] * case["n3"]
    return np.sort(np.random.default_rng([seed, 2]).choice(n, case["n_q"], replace=False)).astype(np.int32) if case["n_q"] else None


def _gamma_in(case, seed):
    n, nb, _ = _modes(case)
    return np.exp(np.random.default_rng([seed, 3]).normal(-4.0, 1.5, size=(5, n * nb)))


def _mesh_of(case):
    return case["n1"], case["n2"], case["n3"]


def prepare(case, seed):
    system = _system(case, seed)
    mesh, prec = _mesh_of(case), fc4.PRECISIONS[case["precision"]]
    s = SimpleNamespace(case=case, system=system, mesh=mesh, precision=prec, q=_subset(case, seed))
    if case["kind"] == "whole":
        return s
    s.engine = fc4.Engine(*system, mesh, precision=prec)
    w, v, e = _harmonic(system[0], system[1], mesh)
    s.engine.set_modes(w.reshape(-1), v.reshape(-1, 3), e)
    if case["sampling"] < 1.0:
        s.engine.set_sampling(case["sampling"], seed)
    if case["kind"] == "kappa":
        s.gamma = torch.from_numpy(_gamma_in(case, seed)).cuda()
        s.dkappa = torch.eye(3, dtype=torch.float64, device="cuda")
    elif case["kind"] == "grad":
        s.phi3, s.phi4 = (torch.from_numpy(p.phi).cuda().requires_grad_() for p in system[2:])
    elif case["kind"] == "bte":
        s.gamma = s.engine.rates(case["T"], case["sigma"], case["mask"], adaptive=case["adaptive"])[0]
    return s


def run(s):
    c = s.case
    T, sg, mask, ad = c["T"], c["sigma"], c["mask"], c["adaptive"]
    if c["kind"] == "kappa":
        return s.engine.kappa(T, s.gamma, mask), s.engine.kappa_backward(T, s.gamma, s.dkappa, mask)
    if c["kind"] == "static":
        return s.engine.rates_static(T, sg, mask, s.q)
    if c["kind"] == "rates":
        return s.engine.rates(T, sg, mask, q_subset=s.q, adaptive=ad)
    if c["kind"] == "bte":
        return s.engine.kappa_iterative(T, sg, s.gamma, mask, adaptive=ad, max_iter=c["iters"], tol=0.0)
    if c["kind"] == "grad":
        gamma = fc4.rates_fn(s.phi3, s.phi4, s.engine, T, sg, mask, adaptive=ad)
        kappa = fc4.kappa_fn(gamma, s.engine, T, mask)
        d3, d4 = torch.autograd.grad(kappa.diagonal().sum(), (s.phi3, s.phi4))
        return gamma.detach(), kappa.detach(), d3, d4
    engine = fc4.Engine(*s.system, s.mesh, precision=s.precision)
    gamma, wp, counts = engine.rates(T, sg, mask, adaptive=ad)
    kappa = engine.kappa(T, gamma, mask)
    engine.close()
    return gamma, wp, counts, kappa


def work(case):
    n, nb, nm = _modes(case)
    nc3, nc4, _ = _clusters(case["atoms"])
    tables = n * nb * (8 + 24 + 16 * nb) + 27 * 8 * nc3 + 81 * 8 * nc4
    if case["kind"] == "kappa":
        return {"bytes": n * nb * (2 * 40 + 32 + 40), "flops": n * nb * 130}
    f = _flops(case)
    if case["kind"] == "grad":
        return {"bytes": 2 * tables + nm * 80, "flops": 3 * f}
    if case["kind"] == "bte":
        return {"bytes": case["iters"] * (tables + nm * 96), "flops": case["iters"] * f}
    if case["kind"] == "whole":
        return {"bytes": 2 * tables + nm * 120, "flops": f + n * 60 * nb ** 3 * 8}
    return {"bytes": tables + nm * 120, "flops": f}


# ------------------------------------------------------------------------------- 64-bit values

def _bose(w, T):
    return torch.where(w > 0, 1.0 / torch.expm1(torch.where(w > 0, w, 1.0) * (HBAR * 1e12 / (KB * T))), 0.0)


def _hash(z):
    """SplitMix64's output function on int64 bit patterns."""
    def shift(x, k):
        return (x >> k) & ((1 << (64 - k)) - 1)
    z = (z ^ shift(z, 30)) * (0xbf58476d1ce4e5b9 - (1 << 64))
    z = (z ^ shift(z, 27)) * (0x94d049bb133111eb - (1 << 64))
    return z ^ shift(z, 31)


class _Dense:
    """Every candidate process of a mode, evaluated densely in FP64."""

    def __init__(self, case, seed, phi3=None, phi4=None):
        self.case, self.seed, self.mesh, self.T = case, seed, _mesh_of(case), case["T"]
        cr, p2, p3, p4 = self.system = _system(case, seed)
        dev = self.dev = torch.device("cuda")
        w, v, e = _harmonic(cr, p2, self.mesh)
        self.w, self.v, self.e = (torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (w, v, e))
        self.n, self.nb = w.shape
        self.na = self.nb // 3
        self.occ = _bose(self.w, self.T)
        self.iw = torch.where(self.w > 0, 1.0 / torch.where(self.w > 0, self.w, 1.0), 0.0)
        self.grid = torch.from_numpy(_grid(self.mesh)).to(dev)
        self.frac = self.grid.double() / torch.tensor(self.mesh, device=dev)
        bx, by, bz = cr.lattice
        recip = 2 * math.pi * np.stack([np.cross(by, bz), np.cross(bz, bx), np.cross(bx, by)]) / np.dot(bx, np.cross(by, bz))
        self.proj = self.v @ torch.from_numpy(recip.T.copy()).to(dev) / torch.tensor(self.mesh, device=dev)
        self.p3 = (p3, torch.from_numpy(p3.phi).to(dev) if phi3 is None else phi3)
        self.p4 = (p4, torch.from_numpy(p4.phi).to(dev) if phi4 is None else phi4)
        self.ism = [torch.from_numpy(1.0 / np.sqrt(np.prod(cr.masses[p.atoms], axis=1))).to(dev) for p in (p3, p4)]
        self.cells = [torch.from_numpy(p.cells.astype(np.float64)).to(dev) for p in (p3, p4)]
        a = p4.atoms
        keys = np.concatenate([a[:, 2:], p4.cells[:, 1] - p4.cells[:, 2]], axis=1)
        self.keys, self.key_of = np.unique(keys, axis=0, return_inverse=True)
        self.key_of = torch.from_numpy(self.key_of.reshape(-1)).to(dev)
        self.pkey = self._phase(self.frac, torch.from_numpy(self.keys[:, 2:].astype(np.float64)).to(dev))

    def _phase(self, frac, cells):
        t = 2 * math.pi * (frac @ cells.T)
        return torch.complex(torch.cos(t), torch.sin(t))

    def _index(self, g):
        g = torch.remainder(g, torch.tensor(self.mesh, device=self.dev))
        return g[..., 0] + self.mesh[0] * (g[..., 1] + self.mesh[1] * g[..., 2])

    def _gauss(self, delta, pa, pb):
        """Weight of the window and the Gaussian; pa, pb: the velocity projections of the width's two legs."""
        if self.case["adaptive"]:
            sg = self.case["sigma"] * torch.sqrt(((pa - pb) ** 2).sum(-1) / 6.0)
        else:
            sg = torch.tensor(2 * math.pi * self.case["sigma"], dtype=torch.float64, device=self.dev)
        keep = (delta.abs() <= 2 * sg) & (sg > 1e-9)
        s = torch.where(sg > 1e-9, sg, 1.0)
        return keep, torch.where(keep, torch.exp(-(delta / s) ** 2) / (s * math.sqrt(math.pi)), 0.0)

    def three(self, ch, q, j):
        """(terms w, |V|², kept, partner indices) over [q', j', j'']."""
        s = 1 if ch == 0 else -1
        (p, phi), ism, cells = self.p3, self.ism[0], self.cells[0]
        q2 = self._index(self.grid[q] + s * self.grid)
        a0 = torch.from_numpy(p.atoms[:, 0].astype(np.int64)).to(self.dev)
        el = self.e[q, :, j].reshape(self.na, 3)[a0]
        A = torch.einsum("nabc,na->nbc", phi.reshape(-1, 3, 3, 3).to(torch.complex128), el) * ism[:, None, None]
        ph = self._phase(s * self.frac, cells[:, 0]) * self._phase(-(self.frac[q] + s * self.frac), cells[:, 1])
        t = torch.zeros(self.na, self.na, self.n, 3, 3, dtype=torch.complex128, device=self.dev)
        rows = []
        for b in range(self.na):
            row = []
            for c in range(self.na):
                k = np.nonzero((p.atoms[:, 1] == b) & (p.atoms[:, 2] == c))[0]
                row.append(torch.einsum("qn,nbc->qbc", ph[:, k], A[k]) if len(k) else t[b, c])
            rows.append(torch.cat(row, dim=2))
        t = torch.cat(rows, dim=1)
        e1 = self.e if s > 0 else self.e.conj()
        V = e1.transpose(1, 2) @ t @ self.e[q2].conj()
        w0, w1, w2 = self.w[q, j], self.w[:, :, None], self.w[q2][:, None, :]
        delta = (w0 + w1) - w2 if ch == 0 else w0 - (w1 + w2)
        keep, g = self._gauss(delta, self.proj[:, :, None], self.proj[q2][:, None, :])
        keep = keep & (w1 > 0) & (w2 > 0)
        n1, n2 = self.occ[:, :, None], self.occ[q2][:, None, :]
        f = n1 - n2 if ch == 0 else 0.5 * (1 + n1 + n2)
        wt = torch.where(keep, f * g * self.iw[q, j] * self.iw[:, :, None] * self.iw[q2][:, None, :], 0.0)
        return wt, V.real ** 2 + V.imag ** 2, keep, (q2,)

    def four(self, ch, q, j):
        """The same over [q', j', q'', j'', j'''], one block of q' at a time."""
        s1, s2 = (-1 if ch == 4 else 1), (1 if ch == 2 else -1)
        (p, phi), ism, cells = self.p4, self.ism[1], self.cells[1]
        at = torch.from_numpy(p.atoms.astype(np.int64)).to(self.dev)
        el = self.e[q, :, j].reshape(self.na, 3)[at[:, 0]]
        B = torch.einsum("nabx,na->nbx", phi.reshape(-1, 3, 3, 9).to(torch.complex128), el) * ism[:, None, None]
        B = B * self._phase(-self.frac[q][None], cells[:, 2])[0][:, None, None]
        e1 = self.e if s1 > 0 else self.e.conj()
        e2 = (self.e if s2 > 0 else self.e.conj()).transpose(1, 2)
        pk = self.pkey if s2 > 0 else self.pkey.conj()
        step = max(1, int(2e7 / (self.n * self.nb ** 3)))
        for lo in range(0, self.n, step):
            k1 = torch.arange(lo, min(self.n, lo + step), device=self.dev)
            b = len(k1)
            ph = self._phase(s1 * self.frac[k1], cells[:, 0] - cells[:, 2])
            e1n = e1[k1].reshape(b, self.na, 3, self.nb)[:, at[:, 1]]
            W = torch.einsum("qn,nbx,qnbj->qjnx", ph, B, e1n)
            W = torch.zeros(b, self.nb, len(self.keys), 9, dtype=W.dtype, device=self.dev).index_add(2, self.key_of, W)
            rows = []
            for c in range(self.na):
                row = []
                for d in range(self.na):
                    r = np.nonzero((self.keys[:, 0] == c) & (self.keys[:, 1] == d))[0]
                    x = torch.einsum("pr,qjrx->qjpx", pk[:, r], W[:, :, r]) if len(r) else \
                        torch.zeros(b, self.nb, self.n, 9, dtype=W.dtype, device=self.dev)
                    row.append(x.reshape(b, self.nb, self.n, 3, 3))
                rows.append(torch.cat(row, dim=4))
            X = torch.cat(rows, dim=3)
            q3 = self._index(self.grid[q] + s1 * self.grid[k1][:, None] + s2 * self.grid[None])
            V = e2 @ X @ self.e[q3].conj()[:, None]
            w0, w1 = self.w[q, j], self.w[k1][:, :, None, None, None]
            w2, w3 = self.w[None, None, :, :, None], self.w[q3][:, None, :, None, :]
            if ch == 2:
                delta = (w0 - w3) + (w1 + w2)
            elif ch == 3:
                delta = (w0 + w1) - (w2 + w3)
            else:
                lo3 = torch.minimum(torch.minimum(w1, w2), w3)
                hi3 = torch.maximum(torch.maximum(w1, w2), w3)
                mid = torch.maximum(torch.minimum(w1, w2), torch.minimum(torch.maximum(w1, w2), w3))
                delta = w0 - ((lo3 + mid) + hi3)
            keep, g = self._gauss(delta, self.proj[None, None, :, :, None, :], self.proj[q3][:, None, :, None, :, :])
            keep = keep & (w1 > 0) & (w2 > 0) & (w3 > 0)
            if self.case["sampling"] < 1.0:
                key = ((q * self.nb + j) * self.n + k1)[:, None] * self.n + torch.arange(self.n, device=self.dev)[None]
                z = _hash(self.seed + (key + 1) * (0x9e3779b97f4a7c15 - (1 << 64)))
                top = int(math.ldexp(self.case["sampling"], 64))
                flip = -(1 << 63)
                keep = keep & ((z ^ flip) < ((top - (1 << 64) if top >= 1 << 63 else top) ^ flip))[:, None, :, None, None]
                g = g * (2.0 ** 64 / top)
            n1, n2 = self.occ[k1][:, :, None, None, None], self.occ[None, None, :, :, None]
            n3 = self.occ[q3][:, None, :, None, :]
            if ch == 2:
                f = 0.5 * (n1 * n2 * (1 + n3) - (1 + n1) * (1 + n2) * n3)
            elif ch == 3:
                f = 0.5 * (n1 * (1 + n2) * (1 + n3) - (1 + n1) * n2 * n3)
            else:
                f = ((1 + n1) * (1 + n2) * (1 + n3) - n1 * n2 * n3) / 6.0
            iw = self.iw[k1][:, :, None, None, None] * self.iw[None, None, :, :, None] * self.iw[q3][:, None, :, None, :]
            yield torch.where(keep, f * g * self.iw[q, j] * iw, 0.0), V.real ** 2 + V.imag ** 2, keep, (k1, q3)

    def mode(self, ch, q, j):
        """Γ (ps⁻¹), WP and kept processes of one channel of mode (q, j)."""
        zero = torch.zeros((), dtype=torch.float64, device=self.dev)
        if q == 0 and j < 3:
            return zero, zero, zero.long()
        if ch < 2:
            wt, v2, keep, _ = self.three(ch, q, j)
            return C3 / self.n * (wt * v2).sum(), wt.sum() / self.n, keep.sum()
        parts = [torch.stack([C4 / self.n ** 2 * (wt * v2).sum(), wt.sum() / self.n ** 2, keep.sum().double()])
                 for wt, v2, keep, _ in self.four(ch, q, j)]
        g, wp, cnt = torch.stack(parts).sum(0)
        return g, wp, cnt.long()

    def rates(self):
        qs = _subset(self.case, self.seed)
        qs = range(self.n) if qs is None else qs.tolist()
        out = [torch.zeros(5, len(qs) * self.nb, dtype=t, device=self.dev) for t in (torch.float64, torch.float64, torch.int64)]
        for ch in range(5):
            if (self.case["mask"] >> ch) & 1:
                for i, (q, j) in enumerate(itertools.product(qs, range(self.nb))):
                    for o, x in zip(out, self.mode(ch, q, j)):
                        o[ch, i] = x
        return out

    def heat(self):
        x = self.w * (HBAR * 1e12 / (KB * self.T))
        scale = 1e-8 / (self.n * abs(np.linalg.det(self.system[0].lattice)) * 1e-30)
        return KB * x * x * self.occ * (self.occ + 1) * scale

    def kappa(self, F):
        return torch.einsum("qj,qjx,qjy->xy", self.heat(), self.v, F)

    def rta(self, gamma):
        g = sum(gamma[ch] for ch in range(5) if (self.case["mask"] >> ch) & 1).reshape(self.n, self.nb)
        ok = (self.w > 0) & (g > 0)
        return torch.where(ok, 1.0 / torch.where(ok, g, 1.0), 0.0)

    def offdiag(self, F):
        """Δ of the iterative Boltzmann equation for the fields F [N, nb, 3]."""
        wf = self.w[..., None] * F
        out = torch.zeros_like(F)
        for q, j in itertools.product(range(self.n), range(self.nb)):
            if q == 0 and j < 3:
                continue
            for ch in (c for c in range(5) if (self.case["mask"] >> c) & 1):
                if ch < 2:
                    wt, v2, _, (q2,) = self.three(ch, q, j)
                    gp = C3 / self.n * wt * v2
                    d = (-1 if ch == 0 else 1) * torch.einsum("qj,qjx->x", gp.sum(2), wf) + torch.einsum("qj,qjx->x", gp.sum(1), wf[q2])
                    out[q, j] += self.iw[q, j] * d
                    continue
                for wt, v2, _, (k1, q3) in self.four(ch, q, j):
                    gp = C4 / self.n ** 2 * wt * v2
                    d = (1 if ch == 4 else -1) * torch.einsum("qj,qjx->x", gp.sum((2, 3, 4)), wf[k1])
                    d += (-1 if ch == 2 else 1) * torch.einsum("pj,pjx->x", gp.sum((0, 1, 4)), wf)
                    d += torch.einsum("qpj,qpjx->x", gp.sum((1, 3)), wf[q3])
                    out[q, j] += self.iw[q, j] * d
        return out


def exact(case, seed):
    n, nb, nm = _modes(case)
    passes = {"bte": case["iters"] + 1, "grad": 4}.get(case["kind"], 1)
    dense = passes * nm * n * n * nb ** 4 if case["mask"] & 28 else 0
    calls = passes * nm * (2 + 3 * (1 + n * n * nb ** 3 // 20_000_000) if case["mask"] & 28 else 2)
    if case["kind"] != "kappa" and (dense > 6e11 or calls > 9000):
        return None
    if case["kind"] == "kappa":
        d = _Dense(case, seed)
        tau = d.rta(torch.from_numpy(_gamma_in(case, seed)).to(d.dev))
        back = -(d.heat() * (d.v ** 2).sum(-1) * tau ** 2).reshape(-1)
        return d.kappa(tau[..., None] * d.v), back[None].expand(5, -1) * torch.tensor([(case["mask"] >> c) & 1 for c in range(5)], device=d.dev)[:, None]
    if case["kind"] in ("static", "rates"):
        return tuple(_Dense(case, seed).rates())
    if case["kind"] == "whole":
        d = _Dense(case, seed)
        gamma, wp, counts = d.rates()
        return None, None, None, d.kappa(d.rta(gamma)[..., None] * d.v)
    if case["kind"] == "bte":
        d = _Dense(case, seed)
        tau = d.rta(d.rates()[0])
        F = tau[..., None] * d.v
        for _ in range(case["iters"]):
            F = tau[..., None] * (d.v + d.offdiag(F))
        return d.kappa(F), F.reshape(-1, 3), case["iters"]
    system = _system(case, seed)
    phi3, phi4 = (torch.from_numpy(p.phi).cuda().requires_grad_() for p in system[2:])
    d = _Dense(case, seed, phi3, phi4)
    with torch.no_grad():
        gamma = d.rates()[0]
        tau = d.rta(gamma)
        slope = -(d.heat() * (d.v ** 2).sum(-1) * tau ** 2)
    d3, d4 = torch.zeros_like(phi3), torch.zeros_like(phi4)
    for ch in (c for c in range(5) if (case["mask"] >> c) & 1):
        for q, j in itertools.product(range(d.n), range(d.nb)):
            if slope[q, j] == 0:
                continue
            terms = [d.three(ch, q, j)] if ch < 2 else d.four(ch, q, j)
            cst = C3 / d.n if ch < 2 else C4 / d.n ** 2
            for wt, v2, _, _ in terms:
                (g,) = torch.autograd.grad(slope[q, j] * cst * (wt * v2).sum(), phi3 if ch < 2 else phi4)
                (d3 if ch < 2 else d4).add_(g)
    return gamma, d.kappa(tau[..., None] * d.v).detach(), d3, d4
