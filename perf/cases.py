"""The work that users of this package have it do, as cases that can be timed.

A case is a dict of plain values; prepare() makes what a program holds before
the call (molecule, basis handle with its Schwarz bounds, density, or a network
and a minibatch), run() is one call of the package's public entry points, and
exact() is the same answer in plain 64-bit torch, from the definitions.

Kinds:
  fock    Basis.fock_build: J and K of one density, the step every SCF iteration repeats
  j       Basis.j_build: J alone
  batch   Batch.fock: J and K of many molecules in one call (CUDA graph)
  scf     Basis.scf: a whole Hartree-Fock calculation
  grad    GuessNet.grad: loss and gradient of one minibatch of the initial-guess network
  forward GuessNet.forward: the network's prediction for one molecule's atom pairs
The seed displaces every atom (thermal motion about the case's geometry) and
draws the density or the minibatch.
"""
import math

import numpy as np
import torch

from fsim_synth import Molecule, Shell, organic_cloud, water, water_cluster
from paper_2510_24968_gb300 import FSIM_DFLOAT, FSIM_FP64, FSIM_MIXED, Basis
from paper_2510_24968_gb300.fsim import Batch
from paper_2510_24968_gb300.guess import NFEAT, NOUT, WIDTH, GuessNet

_PREC = {"fp64": FSIM_FP64, "mixed": FSIM_MIXED, "dfloat": FSIM_DFLOAT}


def _fock(name, mol, n, precision, tau, boys=0.0, spherical=False, fshell=False, kind="fock"):
    case = {"kind": kind, "mol": mol, "n": n, "precision": precision, "tau": tau, "boys": boys,
            "spherical": spherical, "fshell": fshell}
    return {"name": name} | case if name else case


def listed():
    return [
        # one water molecule in FP64, the first thing anyone runs: nothing but launches and latency
        _fock("water_fp64", "water", 1, "fp64", 1e-10),
        # the 152-function water cluster, the size the framework's numbers are quoted on, in each precision
        _fock("water8_mixed", "cluster", 8, "mixed", 1e-10),
        _fock("water8_fp64", "cluster", 8, "fp64", 1e-10),
        _fock("water8_dfloat", "cluster", 8, "dfloat", 1e-10),
        # Coulomb matrix alone
        _fock("water8_j_mixed", "cluster", 8, "mixed", 1e-10, kind="j"),
        # organic-like clouds, rich in p and d: tight threshold; a small one in FP64 (odd, H-capped sizes), a
        # middle one with the Boys function in FP64 accuracy at large T, and the largest case
        _fock("cloud7_fp64", "cloud", 7, "fp64", 1e-11),
        _fock("cloud12_mixed_boys30", "cloud", 12, "mixed", 1e-11, boys=30.0),
        _fock("cloud30_mixed", "cloud", 30, "mixed", 1e-11),
        # f polarisation shells in a spherical basis
        _fock("water3_f_spherical", "cluster", 3, "fp64", 1e-10, spherical=True, fshell=True),
        # many small clusters of uneven size in one call, as training data for the guess is made
        {"name": "batch24_mixed", "kind": "batch", "mol": "cluster", "nmol": 24, "nmin": 2, "nmax": 6,
         "precision": "mixed", "tau": 1e-10},
        # a whole calculation
        {"name": "scf_water5_dfloat", "kind": "scf", "mol": "cluster", "n": 5, "precision": "dfloat", "tau": 1e-10},
        # one training minibatch of the guess network, forward and backward
        {"name": "mlp_grad_4096", "kind": "grad", "batch": 4096},
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fock", "fock", "fock", "fock", "j", "batch", "scf", "f", "grad", "forward"])
    if kind in ("grad", "forward"):
        return {"kind": kind, "batch": _between(rng, 33, 8192)}
    mol = rng.choice(["cluster", "cloud"])
    tau = rng.choice([1e-9, 1e-10, 1e-11, 1e-12])
    if kind == "batch":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        return {"kind": kind, "mol": mol, "nmol": _between(rng, 2, 30 if precision == "mixed" else 7),
                "nmin": rng.randint(1, 3), "nmax": rng.randint(4, 6), "precision": precision, "tau": tau}
    if kind == "scf":
        precision = rng.choice(["dfloat", "fp64"])
        return {"kind": kind, "mol": "cluster", "n": rng.randint(1, 5 if precision == "dfloat" else 3),
                "precision": precision, "tau": rng.choice([1e-10, 1e-11, 1e-12])}
    if kind == "f":
        return _fock("", "cluster", rng.randint(1, 3), rng.choice(["fp64", "mixed"]), tau,
                     spherical=rng.random() < 0.5, fshell=True)
    precision = rng.choice(["mixed", "fp64"] if kind == "j" else ["mixed", "mixed", "fp64", "dfloat"])
    most = {("cluster", "mixed"): 20, ("cloud", "mixed"): 26}.get((mol, precision), 12 if mol == "cluster" else 9)
    return _fock("", mol, _between(rng, 1 if mol == "cluster" else 2, most), precision, tau,
                 boys=rng.choice([0.0, 30.0]) if precision == "mixed" else 0.0, spherical=rng.random() < 0.2 and
                 kind == "fock", kind=kind)


def _molecule(mol, n, seed, fshell=False, geom=1):
    """The case's molecule with every atom displaced by about 0.03 bohr."""
    if mol == "water":
        m = water(0)
    elif mol == "cluster":
        m = water_cluster(n, geom_seed=geom, basis_seed=1)
    else:
        m = organic_cloud(n, geom_seed=geom, basis_seed=2)
    xyz = m.xyz + np.random.default_rng([seed, n, geom]).normal(0.0, 0.03, m.xyz.shape)
    shells = list(m.shells)
    if fshell:
        shells += [Shell(i, 3, (0.6, 1.5, 3.5), (0.8, 0.3, 0.1)) for i, z in enumerate(m.Z) if z > 1]
    return Molecule(m.name, list(m.Z), xyz, shells)


def _molecules(case, seed):
    if case["kind"] != "batch":
        return [_molecule(case["mol"], case["n"], seed, case.get("fshell", False))]
    span = case["nmax"] - case["nmin"] + 1
    return [_molecule(case["mol"], max(case["nmin"] + (5 * i) % span, 2 if case["mol"] == "cloud" else 1), seed, geom=1 + i % 8)
            for i in range(case["nmol"])]


def _density(mol, nbf, seed, per_atom):
    """A symmetric matrix that decays with the distance of its two atoms, as densities do."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    c = torch.tensor(np.asarray(mol.xyz), device="cuda")[torch.tensor(per_atom, device="cuda")]
    near = torch.exp(-torch.cdist(c, c) / 2.5)
    D = torch.randn(nbf, nbf, generator=g, device="cuda", dtype=torch.float64) * near * 0.5
    return (D + D.T).contiguous()


def _atoms_of(mol, spherical):
    return [s.atom for s in mol.shells for _ in range(2 * s.l + 1 if spherical else (s.l + 1) * (s.l + 2) // 2)]


def _minibatch(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    b = case["batch"]
    x = torch.cat([r(b, 16), torch.rand(b, NFEAT - 16, generator=g, device="cuda")], 1)
    t = 0.3 * r(b, NOUT)
    mask = (torch.rand(b, NOUT, generator=g, device="cuda") < 0.45).float()
    p = [r(i * o) / math.sqrt(i) if k == 0 else 0.1 * r(o)
         for i, o in ((NFEAT, WIDTH), (WIDTH, WIDTH), (WIDTH, NOUT)) for k in (0, 1)]
    return x.contiguous(), t.contiguous(), mask.contiguous(), torch.cat(p)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("grad", "forward"):
        x, t, mask, p = _minibatch(case, seed)
        net = GuessNet(params=p.cpu().numpy())
        return {"case": case, "net": net, "x": x, "t": t, "mask": mask,
                "y": torch.zeros(case["batch"], NOUT, device="cuda")}
    mols = _molecules(case, seed)
    sph = case.get("spherical", False)
    bases = [Basis(m, spherical=sph) for m in mols]
    for b in bases:
        b.schwarz()
    s = {"case": case, "bases": bases}
    if kind != "scf":
        s["D"] = [_density(m, b.nbf, seed + 1000 * i, _atoms_of(m, sph)) for i, (m, b) in enumerate(zip(mols, bases))]
        s["J"] = [torch.zeros_like(d) for d in s["D"]]
        s["K"] = [torch.zeros_like(d) for d in s["D"]]
    if kind == "batch":
        s["batch"] = Batch(bases, s["D"], s["J"], s["K"], tau=case["tau"])
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grad":
        loss, g = state["net"].grad(state["x"].data_ptr(), state["t"].data_ptr(), state["mask"].data_ptr(),
                                    case["batch"], bf16=True)
        return {"loss": loss, "grad": g}
    if kind == "forward":
        state["net"].forward(state["x"].data_ptr(), state["y"].data_ptr(), case["batch"])
        return {"y": state["y"]}
    prec = _PREC[case["precision"]]
    if kind == "batch":
        state["batch"].fock(prec)
        return {"J": state["J"], "K": state["K"]}
    b = state["bases"][0]
    if kind == "scf":
        r = b.scf(precision=prec, tau=case["tau"], want_density=True)
        return {"e_total": r["e_total"], "D": r["D"]}
    D, J, K = state["D"][0], state["J"][0], state["K"][0]
    if kind == "j":
        b.j_build(D, J, tau=case["tau"], precision=prec, boys_fp64_T=case["boys"])
        return {"J": J}
    b.fock_build(D, J, K, tau=case["tau"], precision=prec, boys_fp64_T=case["boys"])
    return {"J": J, "K": K}


# ---- the work that a pass cannot do without

def _ncart(l):
    return (l + 1) * (l + 2) // 2


def _nherm(L):
    return (L + 1) * (L + 2) * (L + 3) // 6


def _cart(l):
    return [(a, b, l - a - b) for a in range(l, -1, -1) for b in range(l - a, -1, -1)]


def _nnz(la, lb):
    return sum(np.prod([a[x] + b[x] + 1 for x in range(3)]) for a in _cart(la) for b in _cart(lb))


def _quartet_flops(p, q, npp):
    """Recursion and both transforms of one contracted quartet of npp x npp primitive pairs."""
    (la, lb), (lc, ld) = p, q
    L, A, C = sum(p) + sum(q), _ncart(la) * _ncart(lb), _ncart(lc) * _ncart(ld)
    h1, h2, z1, z2 = _nherm(la + lb), _nherm(lc + ld), _nnz(la, lb), _nnz(lc, ld)
    rec = 2 * sum(_nherm(n) for n in range(L + 1))
    return npp * npp * (rec + min(2 * h1 * z2 + 2 * z1 * C / npp, 2 * h2 * z1 + 2 * z2 * A / npp)) + 12 * A * C


def work(case):
    if case["kind"] in ("grad", "forward"):
        b, w = case["batch"], NFEAT * WIDTH + WIDTH * WIDTH + WIDTH * NOUT
        if case["kind"] == "forward":
            return {"bytes": 4 * b * (NFEAT + NOUT) + 2 * w, "flops": 2 * b * w}
        return {"bytes": 4 * b * (NFEAT + 2 * NOUT) + 2 * w + 4 * w, "flops": 6 * b * w - 2 * b * NFEAT * WIDTH}
    nbytes, flops = 0, 0.0
    for m in _molecules(case, 0):
        b = Basis(m)
        Q, l = b.schwarz(), np.array([s.l for s in m.shells])
        i, j = np.tril_indices(len(l))
        cls = np.maximum(l[i], l[j]) * 4 + np.minimum(l[i], l[j])
        per = {c: np.sort(Q[i, j][cls == c]) for c in np.unique(cls)}
        for x in per:
            for y in per:
                kept = len(per[y]) - np.searchsorted(per[y], case["tau"] / per[x], "left")
                flops += 0.5 * float(kept.sum()) * _quartet_flops(divmod(int(x), 4), divmod(int(y), 4),
                                                                  len(m.shells[0].alpha) ** 2)
        nbytes += 8 * b.nbf ** 2 * (2 if case["kind"] in ("j", "scf") else 3)
    return {"bytes": nbytes, "flops": flops * (17 if case["kind"] == "scf" else 1)}  # an SCF takes about 17 builds


# ---- the same answers in 64 bits, from the definitions (McMurchie-Davidson in dense torch operations)

def _hid(t, u, v):
    n, m = t + u + v, u + v
    return n * (n + 1) * (n + 2) // 6 + m * (m + 1) // 2 + v


def _hermites(L):
    return sorted(((t, u, v) for t in range(L + 1) for u in range(L + 1 - t) for v in range(L + 1 - t - u)),
                  key=lambda h: _hid(*h))


class _Boys:
    """F_0..F_L by an eight-term Taylor expansion of F_L and downward recursion; erf = 1 beyond T = 40."""
    H, TOP, K = 1 / 32, 40.0, 8

    def __init__(self, L):
        T = np.arange(int(self.TOP / self.H) + 2) * self.H
        tab = []
        for m in range(L, L + self.K):
            term = np.full_like(T, 1.0 / (2 * m + 1))
            s = term.copy()
            for i in range(1, 260):
                term = term * 2 * T / (2 * m + 2 * i + 1)
                s += term
            tab.append(np.exp(-T) * s)
        self.L, self.tab = L, torch.tensor(np.array(tab).T.copy(), device="cuda")

    def __call__(self, T):
        big = T >= self.TOP
        Ts = torch.where(big, torch.zeros_like(T), T)
        i = torch.round(Ts / self.H).long()
        x = i * self.H - Ts
        f = self.tab[i, self.K - 1]
        for k in range(self.K - 1, 0, -1):
            f = self.tab[i, k - 1] + f * x / k
        F, e = [f], torch.exp(-Ts)
        for n in range(self.L - 1, -1, -1):
            F.insert(0, (2 * Ts * F[0] + e) / (2 * n + 1))
        if big.any():
            Tb, e = torch.where(big, T, torch.full_like(T, self.TOP)), torch.exp(-T)
            up = [0.5 * torch.sqrt(math.pi / Tb)]
            for n in range(self.L):
                up.append(((2 * n + 1) * up[-1] - e) / (2 * Tb))
            F = [torch.where(big, b, a) for a, b in zip(F, up)]
        return F


def _hermite_R(L, alpha, X, Y, Z, fac, boys):
    """R^0_{tuv} for t+u+v <= L, stacked last."""
    F = boys(alpha * (X * X + Y * Y + Z * Z))
    src = [fac * (-2 * alpha) ** n * F[n] for n in range(L + 1)]
    cur = {(0, 0, 0): src[L]}
    for n in range(L - 1, -1, -1):
        new = {(0, 0, 0): src[n]}
        for h in _hermites(L - n)[1:]:
            x = 0 if h[0] else 1 if h[1] else 2
            lo = tuple(c - (k == x) for k, c in enumerate(h))
            new[h] = (X, Y, Z)[x] * cur[lo]
            if h[x] > 1:
                new[h] = new[h] + (h[x] - 1) * cur[tuple(c - 2 * (k == x) for k, c in enumerate(h))]
        cur = new
    return torch.stack([cur[h] for h in _hermites(L)], -1)


class _Pairs:
    """All shell pairs of two angular momenta: exponents, centres, 1D Hermite coefficients, dense E[pair, prim, comp, hermite]."""

    def __init__(self, mol, sh, la, lb, extra=0):
        ia = [i for i, s in enumerate(mol.shells) if s.l == la]
        ib = [i for i, s in enumerate(mol.shells) if s.l == lb]
        prs = [(i, j) for i in ia for j in ib if la != lb or j <= i]
        dev = dict(device="cuda")
        self.la, self.lb, self.L, self.n = la, lb, la + lb, len(prs)
        A = torch.tensor([p[0] for p in prs], **dev)
        B = torch.tensor([p[1] for p in prs], **dev)
        self.ao = sh["ao"][A], sh["ao"][B]
        self.diff = (A != B).double() + 1.0
        self.shells = A, B
        n = len(prs)
        a = sh["alpha"][A][:, :, None].expand(n, -1, sh["alpha"].shape[1]).reshape(n, -1)
        b = sh["alpha"][B][:, None, :].expand(n, sh["alpha"].shape[1], -1).reshape(n, -1)
        c = (sh["coef"][A][:, :, None] * sh["coef"][B][:, None, :]).reshape(n, -1)
        self.p, self.b = a + b, b
        RA, RB = sh["xyz"][A][:, None, :], sh["xyz"][B][:, None, :]
        self.P = (a[..., None] * RA + b[..., None] * RB) / self.p[..., None]
        self.c = c
        E = {}
        mu, h2 = a * b / self.p, 0.5 / self.p
        for x in range(3):
            PA, PB = self.P[..., x] - RA[..., x], self.P[..., x] - RB[..., x]
            E[x, 0, 0, 0] = torch.exp(-mu * (RA - RB)[..., x] ** 2)
            get = lambda i, j, t: E.get((x, i, j, t)) if 0 <= t <= i + j else None  # noqa: B023,E731
            for i in range(la + 1):
                for j in range(lb + extra + 1):
                    if i == j == 0:
                        continue
                    pi, pj, sft = (i - 1, 0, PA) if j == 0 else (i, j - 1, PB)
                    for t in range(i + j + 1):
                        v = 0
                        for w, k in ((h2, t - 1), (sft, t), (t + 1, t + 1)):
                            e = get(pi, pj, k)
                            if e is not None:
                                v = v + w * e
                        E[x, i, j, t] = v
        self.E1 = E
        comps = [(u, v) for u in _cart(la) for v in _cart(lb)]
        self.norm = [1 / math.sqrt(np.prod([_df(2 * k - 1) for k in u + v])) for u, v in comps]
        self.comps = comps
        Ed = torch.zeros(n, a.shape[1], len(comps), _nherm(self.L), dtype=torch.float64, **dev)
        for k, (u, v) in enumerate(comps):
            for t in range(u[0] + v[0] + 1):
                for m in range(u[1] + v[1] + 1):
                    for w in range(u[2] + v[2] + 1):
                        Ed[:, :, k, _hid(t, m, w)] = self.norm[k] * c * E[0, u[0], v[0], t] * E[1, u[1], v[1], m] * E[2, u[2], v[2], w]
        self.E = Ed


def _df(n):
    return math.prod(range(n, 0, -2)) if n > 0 else 1


def _shell_data(mol):
    npr = max(len(s.alpha) for s in mol.shells)
    al, co, xyz, ao, k = [], [], [], [], 0
    for s in mol.shells:
        a, d = np.array(s.alpha), np.array(s.coef)
        d = d * (2 * a / math.pi) ** 0.75 * (4 * a) ** (s.l / 2)
        ov = np.sum(np.outer(d, d) * (math.pi / np.add.outer(a, a)) ** 1.5 / (2 * np.add.outer(a, a)) ** s.l)
        al.append(np.concatenate([a, np.ones(npr - len(a))]))
        co.append(np.concatenate([d / math.sqrt(ov), np.zeros(npr - len(a))]))
        xyz.append(mol.xyz[s.atom])
        ao.append(k)
        k += _ncart(s.l)
    d = {k: torch.tensor(np.array(v), device="cuda", dtype=torch.float64) for k, v in (("alpha", al), ("coef", co), ("xyz", xyz))}
    return d | {"ao": torch.tensor(ao, device="cuda"), "nbf": k}


class _Integrals:
    def __init__(self, mol, tau):
        self.mol, self.sh, self.tau = mol, _shell_data(mol), tau
        ls = sorted({s.l for s in mol.shells})
        self.cls = [_Pairs(mol, self.sh, a, b) for a in ls for b in ls if b <= a]
        self.boys, self.Q = {}, []
        for p in self.cls:
            i = torch.arange(p.n, device="cuda")
            q = [torch.diagonal(g, dim1=1, dim2=2).abs().amax(1) for _, _, g in self.blocks(p, p, i, i)]
            self.Q.append(torch.sqrt(torch.cat(q)))
        # screened unique quartets of each class pair
        self.lists = []
        for x, p in enumerate(self.cls):
            for y, q in enumerate(self.cls[:x + 1]):
                keep = torch.outer(self.Q[x], self.Q[y]) >= tau
                i, j = torch.nonzero(torch.tril(keep) if x == y else keep, as_tuple=True)
                self.lists.append((p, q, i, j, x == y))

    def blocks(self, p, q, i, j):
        """(i, j, (ab|cd) blocks [quartet, a, c]) for bra pairs i and ket pairs j, in chunks."""
        L = p.L + q.L
        if L not in self.boys:
            self.boys[L] = _Boys(L)
        boys = self.boys[L]
        hb, hk = _hermites(p.L), _hermites(q.L)
        where = torch.tensor([[_hid(*(a + b for a, b in zip(u, v))) for v in hk] for u in hb], device="cuda")
        sign = torch.tensor([(-1.0) ** sum(v) for v in hk], device="cuda", dtype=torch.float64)
        kb, kk = p.p.shape[1], q.p.shape[1]
        step = max(1, int(1.5e8 / (kb * kk * max(len(hb) * len(hk), 3 * _nherm(L)))))
        for c in range(0, len(i), step):
            ii, jj = i[c:c + step], j[c:c + step]
            pp, qq = p.p[ii][:, :, None], q.p[jj][:, None, :]
            d = p.P[ii][:, :, None, :] - q.P[jj][:, None, :, :]
            R = _hermite_R(L, pp * qq / (pp + qq), d[..., 0], d[..., 1], d[..., 2],
                           2 * math.pi ** 2.5 / (pp * qq * torch.sqrt(pp + qq)), boys)
            R = R[..., where] * sign                                       # [q, b, k, h, h']
            n = len(ii)
            M = R.permute(0, 1, 3, 2, 4).reshape(n, kb * len(hb), kk * len(hk))
            W = torch.bmm(M, q.E[jj].permute(0, 1, 3, 2).reshape(n, kk * len(hk), -1))
            yield ii, jj, torch.bmm(p.E[ii].permute(0, 2, 1, 3).reshape(n, -1, kb * len(hb)), W)

    def jk(self, D):
        N = self.sh["nbf"]
        J, K = (torch.zeros(N * N, dtype=torch.float64, device="cuda") for _ in range(2))
        ar = lambda l: torch.arange(_ncart(l), device="cuda")  # noqa: E731
        for p, q, i, j, same in self.lists:
            for ii, jj, g in self.blocks(p, q, i, j):
                deg = p.diff[ii] * q.diff[jj] * (torch.where(ii == jj, 1.0, 2.0) if same else 2.0)
                v = (g * deg[:, None, None].double()).reshape(len(ii), _ncart(p.la), _ncart(p.lb), _ncart(q.la), _ncart(q.lb))
                m, n = p.ao[0][ii][:, None] + ar(p.la), p.ao[1][ii][:, None] + ar(p.lb)
                l, s = q.ao[0][jj][:, None] + ar(q.la), q.ao[1][jj][:, None] + ar(q.lb)
                at = lambda r, c: (r[:, :, None] * N + c[:, None, :])  # noqa: E731
                for out, eq, src, dst in ((J, "zmnls,zmn->zls", at(m, n), at(l, s)), (J, "zmnls,zls->zmn", at(l, s), at(m, n)),
                                          (K, "zmnls,zns->zml", at(n, s), at(m, l)), (K, "zmnls,zml->zns", at(m, l), at(n, s)),
                                          (K, "zmnls,znl->zms", at(n, l), at(m, s)), (K, "zmnls,zms->znl", at(m, s), at(n, l))):
                    out.index_add_(0, dst.reshape(-1), torch.einsum(eq, v, D.reshape(-1)[src]).reshape(-1))
        J, K = J.reshape(N, N), K.reshape(N, N)
        return (J + J.T) / 4, (K + K.T) / 8

    def one_electron(self):
        """Overlap and kinetic energy plus nuclear attraction."""
        N, mol = self.sh["nbf"], self.mol
        S, H = (torch.zeros(N, N, dtype=torch.float64, device="cuda") for _ in range(2))
        for c in self.cls:
            p = _Pairs(mol, self.sh, c.la, c.lb, extra=2)
            Vh = 0
            boys = _Boys(p.L)
            for Z, R in zip(mol.Z, mol.xyz):
                d = p.P - torch.tensor(R, device="cuda")
                Vh = Vh - Z * _hermite_R(p.L, p.p, d[..., 0], d[..., 1], d[..., 2], 2 * math.pi / p.p, boys)
            V = torch.einsum("zkch,zkh->zc", p.E, Vh)
            root = torch.sqrt(math.pi / p.p)
            o = lambda x, i, j: p.E1[x, i, j, 0] * root if j >= 0 else 0.0  # noqa: B023,E731
            kin = lambda x, i, j: -0.5 * (4 * p.b ** 2 * o(x, i, j + 2) - 2 * p.b * (2 * j + 1) * o(x, i, j) + j * (j - 1) * o(x, i, j - 2))  # noqa: B023,E731,E501
            for k, (u, v) in enumerate(p.comps):
                f = [(o(x, u[x], v[x]), kin(x, u[x], v[x])) for x in range(3)]
                w = p.norm[k] * p.c
                s = (w * f[0][0] * f[1][0] * f[2][0]).sum(1)
                t = (w * (f[0][1] * f[1][0] * f[2][0] + f[0][0] * f[1][1] * f[2][0] + f[0][0] * f[1][0] * f[2][1])).sum(1)
                r, q = p.ao[0] + k // _ncart(p.lb), p.ao[1] + k % _ncart(p.lb)
                S[r, q] = S[q, r] = s
                H[r, q] = H[q, r] = t + V[:, k]
        return S, H


def _solid(l):
    """Rows: the 2l+1 real solid harmonics on the unit-normalised Cartesian components."""
    if l < 2:
        return np.eye(_ncart(l))
    poly = {2: [{(1, 1, 0): 1}, {(0, 1, 1): 1}, {(0, 0, 2): 2, (2, 0, 0): -1, (0, 2, 0): -1}, {(1, 0, 1): 1},
                {(2, 0, 0): 1, (0, 2, 0): -1}],
            3: [{(2, 1, 0): 3, (0, 3, 0): -1}, {(1, 1, 1): 1}, {(0, 1, 2): 4, (2, 1, 0): -1, (0, 3, 0): -1},
                {(0, 0, 3): 2, (2, 0, 1): -3, (0, 2, 1): -3}, {(1, 0, 2): 4, (3, 0, 0): -1, (1, 2, 0): -1},
                {(2, 0, 1): 1, (0, 2, 1): -1}, {(3, 0, 0): 1, (1, 2, 0): -3}]}[l]
    cart = _cart(l)
    root = [math.sqrt(np.prod([_df(2 * k - 1) for k in c])) for c in cart]
    ov = np.array([[0.0 if any((x + y) % 2 for x, y in zip(a, b)) else np.prod([_df(x + y - 1) for x, y in zip(a, b)])
                    for b in cart] for a in cart]) / np.outer(root, root)
    rows = np.array([[r.get(c, 0) * w for c, w in zip(cart, root)] for r in poly])
    return rows / np.sqrt(np.einsum("ia,ab,ib->i", rows, ov, rows))[:, None]


def _exact_jk(mol, tau, D, spherical):
    g = _Integrals(mol, tau)
    if not spherical:
        return g.jk(D)
    T = torch.block_diag(*[torch.tensor(_solid(s.l), device="cuda") for s in mol.shells])
    J, K = g.jk(T.T @ D @ T)
    return T @ J @ T.T, T @ K @ T.T


def _exact_scf(mol, tau):
    """Restricted Hartree-Fock with DIIS to far below the calculation's own thresholds."""
    g = _Integrals(mol, tau)
    S, H = g.one_electron()
    w, U = torch.linalg.eigh(S)
    X = U @ torch.diag(w ** -0.5) @ U.T
    nocc, Fs, es, enuc = mol.nelec // 2, [], [], 0.0
    for a in range(mol.natom):
        for b in range(a):
            enuc += mol.Z[a] * mol.Z[b] / float(np.linalg.norm(mol.xyz[a] - mol.xyz[b]))
    F, D, E = H, None, 0.0
    for _ in range(80):
        C = X @ torch.linalg.eigh(X.T @ F @ X)[1][:, :nocc]
        new = 2 * C @ C.T
        moved = math.inf if D is None else float((new - D).square().mean().sqrt())
        D = new
        J, K = g.jk(D)
        F = H + J - 0.5 * K
        E = 0.5 * float((D * (H + F)).sum())
        if moved < 1e-10:
            break
        e = F @ D @ S
        Fs, es = (Fs + [F])[-8:], (es + [e - e.T])[-8:]
        if len(Fs) > 1:
            n = len(Fs)
            B = torch.full((n + 1, n + 1), -1.0, dtype=torch.float64)
            B[n, n] = 0.0
            B[:n, :n] = torch.tensor([[float((x * y).sum()) for y in es] for x in es])
            rhs = torch.zeros(n + 1, dtype=torch.float64)
            rhs[n] = -1.0
            F = sum(float(k) * f for k, f in zip(torch.linalg.solve(B, rhs), Fs))
    return {"e_total": torch.tensor(E + enuc, dtype=torch.float64), "D": D}


def _exact_net(case, seed):
    x, t, mask, p = (v.double() for v in _minibatch(case, seed))
    p = p.clone().requires_grad_()
    k, y = 0, x
    for n, (i, o) in enumerate(((NFEAT, WIDTH), (WIDTH, WIDTH), (WIDTH, NOUT))):
        y = y @ p[k:k + i * o].reshape(i, o) + p[k + i * o:k + i * o + o]
        y = torch.nn.functional.silu(y) if n < 2 else y
        k += i * o + o
    if case["kind"] == "forward":
        return {"y": y.detach()}
    loss = (mask * (y - t) ** 2).sum() / mask.sum()
    loss.backward()
    return {"loss": loss.detach(), "grad": p.grad}


def exact(case, seed):
    if case["kind"] in ("grad", "forward"):
        return _exact_net(case, seed)
    mols = _molecules(case, seed)
    if case["mol"] == "cloud" and max(m.natom for m in mols) > 13:
        return None  # minutes
    if case["kind"] == "scf":
        return _exact_scf(mols[0], case["tau"])
    sph, Js, Ks = case.get("spherical", False), [], []
    for i, m in enumerate(mols):
        atoms = _atoms_of(m, sph)
        J, K = _exact_jk(m, case["tau"], _density(m, len(atoms), seed + 1000 * i, atoms), sph)
        Js.append(J)
        Ks.append(K)
    if case["kind"] == "batch":
        return {"J": Js, "K": Ks}
    return {"J": Js[0]} if case["kind"] == "j" else {"J": Js[0], "K": Ks[0]}
