"""The work that is timed: what a user of this package has it do, case by case.

A case names a kind of call, a molecule and the options of the call.  The
molecule's composition (elements, shells, exponents, contraction
coefficients) comes from the case alone; the seed moves every atom a little,
as a step of a geometry optimisation does, and draws the density or the
orbitals.  Kinds:

  jk      Coulomb and exchange matrices of one density (one Fock build)
  ujk     the same of two spin densities from one integral evaluation
  grad    analytic nuclear gradient from given orbitals
  stored  the dense integral tensor, then J and K from it
  mp2     second-order correlation energy from given orbitals
  scf     a new molecule: basis set-up, then a fixed number of RHF iterations
  batch   several new molecules: basis set-up, then batched RHF iterations

Basis rules: "s" one contracted s shell per atom on a line; "sp" and "spd"
lattice molecules of H, C and O (2 s shells on H, 3 s + 2 p on C and O, with
"spd" one d shell more and 1 to 6 primitives a shell instead of 3); "qz" one
water molecule, or its first one or two atoms, in a basis of quadruple-zeta
shape up to g.
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1303_4916_gb300 as hf

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # the smallest call: a minimal chain of eight hydrogens, a few thousand primitive quartets, all latency
        dict(name="jk_h8_fp64", kind="jk", rules="s", natom=8, mol_seed=0, tier="fp64"),
        # the everyday Fock build in the default precision: 40 atoms, s and p shells (the size of the headline benchmark)
        dict(name="jk_sp40_fp64", kind="jk", rules="sp", natom=40, mol_seed=1, tier="fp64"),
        # the same build in the double-float tier, which long runs choose
        dict(name="jk_sp40_df64", kind="jk", rules="sp", natom=40, mol_seed=1, tier="df64"),
        # a small molecule with d shells and ragged contractions: classes that the lattice of s and p shells does not have
        dict(name="jk_spd9_fp64", kind="jk", rules="spd", natom=9, mol_seed=3, tier="fp64"),
        # a larger one in the mixed tier (double-float, small quartets in FP32), the fastest that the package offers
        dict(name="jk_spd20_mixed", kind="jk", rules="spd", natom=20, mol_seed=5, tier="mixed"),
        # f and g shells: water in a quadruple-zeta basis, 140 functions
        dict(name="jk_qz3_fp64", kind="jk", rules="qz", natom=3, mol_seed=0, tier="fp64"),
        # an open shell: two spin densities, odd atom count
        dict(name="ujk_sp15_fp64", kind="ujk", rules="sp", natom=15, mol_seed=7, tier="fp64"),
        # forces on the water molecule
        dict(name="grad_qz3", kind="grad", rules="qz", natom=3, mol_seed=0, tier="fp64"),
        # forces on a molecule of s, p and d shells
        dict(name="grad_spd5", kind="grad", rules="spd", natom=5, mol_seed=2, tier="fp64"),
        # a small molecule kept in memory: the tensor once, and a contraction with it
        dict(name="stored_spd11", kind="stored", rules="spd", natom=11, mol_seed=4, tier="fp64"),
        # whole calls: a new molecule through set-up and ten iterations; six molecules at once
        dict(name="scf_sp7", kind="scf", rules="sp", natom=7, mol_seed=6, tier="fp64"),
        dict(name="batch6_sp4", kind="batch", rules="sp", natom=4, mol_seed=20, tier="df64"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["jk", "jk", "jk", "jk", "ujk", "grad", "stored", "mp2", "scf", "batch"])
    rules = rng.choice({"jk": ["s", "sp", "sp", "spd", "spd", "qz"], "ujk": ["sp", "spd", "qz"], "grad": ["sp", "spd", "qz"],
                        "stored": ["sp", "spd"], "mp2": ["sp", "spd"], "scf": ["s", "sp"], "batch": ["s", "sp"]}[kind])
    lo, hi = {"jk": {"s": (2, 64), "sp": (3, 32), "spd": (2, 12), "qz": (1, 3)}, "ujk": {"sp": (3, 25), "spd": (2, 8), "qz": (1, 3)},
              "grad": {"sp": (3, 7), "spd": (2, 5), "qz": (1, 3)}, "stored": {"sp": (3, 20), "spd": (2, 9)}, "mp2": {"sp": (4, 14), "spd": (3, 7)},
              "scf": {"s": (4, 32), "sp": (3, 10)}, "batch": {"s": (4, 16), "sp": (3, 7)}}[kind][rules]
    # the gradient, the stored tensor, MP2 and RHF by itself have no tiers
    tier = rng.choice(["fp64", "df64", "mixed"]) if kind in ("jk", "ujk", "batch") else "fp64"
    return dict(kind=kind, rules=rules, natom=size(lo, hi), mol_seed=rng.randrange(100, 10000), tier=tier)


# ---------------------------------------------------------------- molecules

_SHELLS = {"s": {1: [0]}, "sp": {1: [0, 0], 6: [0, 0, 0, 1, 1], 8: [0, 0, 0, 1, 1]},
           "spd": {1: [0, 0], 6: [0, 0, 0, 1, 1, 2], 8: [0, 0, 0, 1, 1, 2]}}
_NPRIM = {"s": (3, 3), "sp": (3, 3), "spd": (1, 6)}
_EXPS = {"s": (0.1, 10.0), "sp": (0.05, 50.0), "spd": (0.03, 200.0)}
# quadruple-zeta shape: (l, primitives) per shell, and the exponent range of each l
_QZ = {8: [(0, 12), (0, 12), (0, 1), (0, 1), (0, 1), (1, 6), (1, 1), (1, 1), (1, 1), (2, 1), (2, 1), (2, 1), (3, 1), (3, 1), (4, 1)],
       1: [(0, 4), (0, 1), (0, 1), (0, 1), (1, 1), (1, 1), (1, 1), (2, 1), (2, 1), (3, 1)]}
_QZ_EXP = {8: {0: (0.1, 6.0e4), 1: (0.1, 60.0), 2: (0.3, 4.0), 3: (0.5, 3.0), 4: (1.0, 2.5)},
           1: {0: (0.05, 80.0), 1: (0.2, 3.0), 2: (0.5, 2.5), 3: (0.8, 1.5)}}


def _molecule(rules, natom, mol_seed, seed):
    """Elements, shells and the reference geometry from mol_seed; the seed moves every atom by up to 0.03 bohr."""
    rng = np.random.default_rng([77, mol_seed])
    if rules == "s":
        Z = np.ones(natom, dtype=np.int32)
        xyz = np.stack([1.4 * np.arange(natom), np.zeros(natom), np.zeros(natom)], axis=1) + rng.uniform(-0.1, 0.1, (natom, 3))
    elif rules == "qz":
        half, r = math.radians(104.5) / 2, 1.809
        Z = np.array([8, 1, 1], dtype=np.int32)[:natom]
        xyz = np.array([[0, 0, 0], [r * math.sin(half), r * math.cos(half), 0], [-r * math.sin(half), r * math.cos(half), 0]])[:natom]
    else:
        n = 1
        while n ** 3 < natom:
            n += 1
        sites = np.array([(i, j, k) for i in range(n) for j in range(n) for k in range(n)][:natom], dtype=float)
        xyz = 2.4 * sites + rng.uniform(-0.3, 0.3, (natom, 3))
        Z = rng.choice([1, 6, 8], size=natom, p=[0.5, 0.3, 0.2]).astype(np.int32)
    shells = []
    for a in range(natom):
        if rules == "qz":
            spec = _QZ[int(Z[a])]
            for l in sorted({x for x, _ in spec}):
                lo, hi = _QZ_EXP[int(Z[a])][l]
                single = sum(1 for x, k in spec if x == l and k == 1)
                for x, k in spec:
                    if x == l and k > 1:
                        shells.append((a, l, np.exp(rng.uniform(math.log(lo), math.log(hi), k)), rng.uniform(0.2, 1.0, k)))
                for i in range(single):
                    t = (i + 0.5 + rng.uniform(-0.2, 0.2)) / single
                    shells.append((a, l, np.array([lo * (hi / lo) ** t]), np.ones(1)))
        else:
            for l in _SHELLS[rules][int(Z[a])]:
                k = int(rng.integers(_NPRIM[rules][0], _NPRIM[rules][1] + 1))
                lo, hi = _EXPS[rules]
                shells.append((a, l, np.exp(rng.uniform(math.log(lo), math.log(hi), k)), rng.uniform(0.2, 1.0, k)))
    if seed is not None:
        xyz = xyz + np.random.default_rng([78, mol_seed, seed]).uniform(-0.03, 0.03, (natom, 3))
    count = np.array([len(s[2]) for s in shells])
    ls = np.array([s[1] for s in shells], dtype=np.int32)
    return SimpleNamespace(Z=Z, xyz=np.ascontiguousarray(xyz, dtype=np.float64), shell_atom=np.array([s[0] for s in shells], dtype=np.int32), shell_l=ls,
                           shell_nprim=count.astype(np.int32), shell_prim=(np.cumsum(count) - count).astype(np.int32),
                           exps=np.concatenate([s[2] for s in shells]), coefs=np.concatenate([s[3] for s in shells]),
                           n_electrons=int(Z.sum()) // 2 * 2, nbf=int(((ls + 1) * (ls + 2) // 2).sum()))


def _molecules(case, seed):
    if case["kind"] == "batch":  # sizes natom .. natom + 5
        return [_molecule(case["rules"], case["natom"] + i, case["mol_seed"] + i, seed) for i in range(6)]
    return [_molecule(case["rules"], case["natom"], case["mol_seed"], seed)]


def _density(n, nocc, seed, k):
    c = np.random.default_rng([79, seed, k]).normal(size=(n, nocc)) / math.sqrt(n)
    return c @ c.T


def _orbitals(n, seed):
    """Orthonormal columns and ascending energies with a gap, as a converged calculation hands them on."""
    rng = np.random.default_rng([80, seed])
    c, _ = np.linalg.qr(rng.normal(size=(n, n)))
    return c / math.sqrt(n)


def _energies(n, nocc, seed):
    rng = np.random.default_rng([81, seed])
    return np.concatenate([np.sort(rng.uniform(-20.0, -0.4, nocc)), np.sort(rng.uniform(0.2, 6.0, n - nocc))])


# ---------------------------------------------------------------- the calls


@functools.lru_cache(maxsize=1)
def _context():
    return hf.Context(0)


def _tier(tier):
    return {"fp64": {}, "df64": dict(df64=True), "mixed": dict(df64=True, fp32_bound=1e-5)}[tier]


def prepare(case, seed):
    mols = _molecules(case, seed)
    mol, kind = mols[0], case["kind"]
    s = SimpleNamespace(kind=kind, ctx=_context(), mols=mols, tier=_tier(case["tier"]), nocc=max(1, mol.n_electrons // 2))
    if kind in ("scf", "batch"):
        return s
    s.basis = hf.Basis(s.ctx, mol)
    n = mol.nbf
    if kind in ("jk", "ujk", "stored"):
        s.D = torch.tensor(_density(n, s.nocc, seed, 0), device="cuda")
        s.D2 = torch.tensor(_density(n, max(1, s.nocc - 1), seed, 1), device="cuda")
        s.opts = hf.jk_opts(1e-12, **s.tier)
    else:
        s.nocc = min(s.nocc, n - 1)
        s.C = torch.tensor(_orbitals(n, seed), device="cuda")
        s.eps = torch.tensor(_energies(n, s.nocc, seed), device="cuda")
        s.result = SimpleNamespace(tensors=dict(C=s.C, eps=s.eps))
    return s


def run(s):
    if s.kind == "jk":
        return s.basis.fock_jk(s.D, opts=s.opts)
    if s.kind == "ujk":
        return s.basis.fock_jk_uhf(s.D, s.D2, opts=s.opts)
    if s.kind == "grad":
        return s.basis.gradient(s.result)
    if s.kind == "stored":
        g = s.basis.eri_tensor()
        j, k = s.basis.jk_stored(g, s.D)
        return g, j, k
    if s.kind == "mp2":
        return s.basis.mp2_energy(s.C, s.eps, s.nocc)
    # ten iterations, which is before the stopping rule takes hold: a count that a change of the last bit does not move
    if s.kind == "scf":
        r = hf.Basis(s.ctx, s.mols[0]).scf(max_iter=10, e_tol=1e-13)
        return dict(energy=r.energy, D=r.tensors["D"], F=r.tensors["F"], eps=r.tensors["eps"])
    res, _ = hf.scf_solve_batch([hf.Basis(s.ctx, m) for m in s.mols], max_iter=10, e_tol=1e-13, **s.tier)
    return np.array([r.energy for r in res])


# ---------------------------------------------------------------- floors


def _pair_counts(mol):
    """Per pair class (la, lb): shell pairs, and primitive pairs whose overlap factor is not negligible."""
    out = {}
    xyz = mol.xyz[mol.shell_atom]
    for i in range(len(mol.shell_l)):
        ei = mol.exps[mol.shell_prim[i]:mol.shell_prim[i] + mol.shell_nprim[i]]
        for j in range(i + 1):
            ej = mol.exps[mol.shell_prim[j]:mol.shell_prim[j] + mol.shell_nprim[j]]
            r2 = float(((xyz[i] - xyz[j]) ** 2).sum())
            live = int((np.outer(ei, ej) / np.add.outer(ei, ej) * r2 < 39.0).sum())
            key = tuple(sorted((int(mol.shell_l[i]), int(mol.shell_l[j])), reverse=True))
            a, b = out.get(key, (0, 0))
            out[key] = (a + (live > 0), b + live)
    return sorted(out.items())


def _nc(l):
    return (l + 1) * (l + 2) // 2


def _integral_flops(mol, digest, derivative):
    """Operations of one pass over the unique quartets: per primitive quartet the set-up and F_m (about 40) and one multiply-add for each
    [e0|f0] that the contraction needs; per shell quartet the contraction of the block with the density (`digest` per integral)."""
    cls = _pair_counts(mol)
    total = 0.0
    for x, (bra, (nb, pb)) in enumerate(cls):
        for y in range(x + 1):
            ket, (nk, pk) = cls[y]
            half = 0.5 if x == y else 1.0
            ne = sum(_nc(l) for l in range(bra[0], bra[0] + bra[1] + 1 + derivative))
            nf = sum(_nc(l) for l in range(ket[0], ket[0] + ket[1] + 1 + derivative))
            block = _nc(bra[0]) * _nc(bra[1]) * _nc(ket[0]) * _nc(ket[1])
            total += half * (pb * pk * (40.0 + 2.0 * ne * nf) + nb * nk * digest * block)
    return total


def work(case):
    total = {"bytes": 0.0, "flops": 0.0}
    for mol in _molecules(case, None):
        n, kind = mol.nbf, case["kind"]
        nocc = max(1, min(mol.n_electrons // 2, n - 1))
        if kind in ("jk", "ujk"):
            b, f = (3 if kind == "jk" else 5) * 8.0 * n * n, _integral_flops(mol, 12 if kind == "jk" else 20, 0)
        elif kind == "grad":
            b, f = 8.0 * n * n, _integral_flops(mol, 18, 1)
        elif kind == "stored":  # the tensor written, then read once for both contractions
            b, f = 2 * 8.0 * n ** 4, _integral_flops(mol, 0, 0) + 4.0 * n ** 4
        elif kind == "mp2":
            nv = n - nocc
            b, f = 8.0 * n * n, _integral_flops(mol, 0, 0) + 2.0 * nocc * (n ** 4 + n ** 3 * nv + n * n * nocc * nv + n * nocc * nv * nv) + 6.0 * (nocc * nv) ** 2
        else:  # ten iterations: a build, five products and an eigenproblem each
            b, f = 10 * 4 * 8.0 * n * n, 10 * (_integral_flops(mol, 12, 0) + 10.0 * n ** 3 + 9.0 * n ** 3)
        total["bytes"] += b
        total["flops"] += f
    return total


# ---------------------------------------------------------------- 64-bit values
# The integrals by the McMurchie-Davidson scheme (Hermite Gaussians), in plain float64 torch, no screening.


def _comps(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _df(n):
    return math.prod(range(n, 0, -2)) if n > 0 else 1


def _herm(L):
    return [(t, u, v) for t in range(L + 1) for u in range(L + 1 - t) for v in range(L + 1 - t - u)]


def _boys(M, T):
    """F_0 .. F_M: below 35 the ascending series of F_M and downward recursion, above it upward recursion from F_0."""
    small = T < 35.0
    t, e = torch.where(small, T, torch.zeros_like(T)), torch.exp(-T)
    term = torch.full_like(T, 1.0 / (2 * M + 1))
    acc = term.clone()
    for i in range(1, 150):
        term = term * (2.0 * t / (2 * M + 2 * i + 1))
        acc += term
    F = [None] * (M + 1)
    F[M] = acc * e
    for m in range(M - 1, -1, -1):
        F[m] = (2.0 * t * F[m + 1] + e) / (2 * m + 1)
    big = torch.where(small, torch.full_like(T, 35.0), T)
    up = 0.5 * torch.sqrt(math.pi / big) * torch.erf(torch.sqrt(big))
    for m in range(M + 1):
        F[m] = torch.where(small, F[m], up)
        up = ((2 * m + 1) * up - e) / (2.0 * big)
    return F


def _exact_pairs(mol, dev):
    """Per pair class: function indices [pairs, na, nb], exponents p and centres P of the (padded) primitive pairs, Hermite coefficients."""
    norm = []
    for s in range(len(mol.shell_l)):
        l, sl = int(mol.shell_l[s]), slice(mol.shell_prim[s], mol.shell_prim[s] + mol.shell_nprim[s])
        e = mol.exps[sl]
        c = mol.coefs[sl] * (2 * e / math.pi) ** 0.75 * (4 * e) ** (l / 2) / math.sqrt(_df(2 * l - 1))
        p = np.add.outer(e, e)
        norm.append(c / math.sqrt((np.outer(c, c) * (math.pi / p) ** 1.5 * _df(2 * l - 1) / (2 * p) ** l).sum()))
    off = np.concatenate([[0], np.cumsum([_nc(int(l)) for l in mol.shell_l])])
    groups = {}
    for i in range(len(mol.shell_l)):
        for j in range(i + 1):
            a, b = (i, j) if mol.shell_l[i] >= mol.shell_l[j] else (j, i)
            groups.setdefault((int(mol.shell_l[a]), int(mol.shell_l[b])), []).append((a, b))
    out = []
    for (la, lb), pairs in sorted(groups.items()):
        width = max(int(mol.shell_nprim[a]) * int(mol.shell_nprim[b]) for a, b in pairs)
        ea, eb, cc = np.ones((len(pairs), width)), np.ones((len(pairs), width)), np.zeros((len(pairs), width))
        A, B = np.zeros((len(pairs), 3)), np.zeros((len(pairs), 3))
        for r, (a, b) in enumerate(pairs):
            xa, xb = (mol.exps[mol.shell_prim[s]:mol.shell_prim[s] + mol.shell_nprim[s]] for s in (a, b))
            k = len(xa) * len(xb)
            ea[r, :k], eb[r, :k], cc[r, :k] = np.repeat(xa, len(xb)), np.tile(xb, len(xa)), np.outer(norm[a], norm[b]).ravel()
            A[r], B[r] = mol.xyz[mol.shell_atom[a]], mol.xyz[mol.shell_atom[b]]
        ea, eb, cc, A, B = (torch.tensor(v, device=dev) for v in (ea, eb, cc, A, B))
        p = ea + eb
        P = (ea[..., None] * A[:, None] + eb[..., None] * B[:, None]) / p[..., None]
        E = []
        for x in range(3):
            d = (A[:, x] - B[:, x])[:, None]
            pa, pb = P[..., x] - A[:, None, x], P[..., x] - B[:, None, x]
            tab = {(0, 0, 0): torch.exp(-ea * eb / p * d * d)}
            get = lambda i, j, t: tab.get((i, j, t), 0.0)  # noqa: E731
            for i in range(la + 1):
                for j in range(lb + 1):
                    if i + j == 0:
                        continue
                    for t in range(i + j + 1):
                        u, v, w = ((i - 1, j), pa, t) if i > 0 else ((i, j - 1), pb, t)
                        tab[(i, j, t)] = get(*u, w - 1) / (2 * p) + v * get(*u, w) + (w + 1) * get(*u, w + 1)
            E.append(tab)
        herm = _herm(la + lb)
        H = torch.zeros((len(pairs), width, _nc(la) * _nc(lb), len(herm)), dtype=torch.float64, device=dev)
        zero = torch.zeros_like(p)
        for ia, ca in enumerate(_comps(la)):
            for ib, cb in enumerate(_comps(lb)):
                scale = math.sqrt(_df(2 * la - 1) / math.prod(_df(2 * k - 1) for k in ca)) * math.sqrt(_df(2 * lb - 1) / math.prod(_df(2 * k - 1) for k in cb))
                for h, q in enumerate(herm):
                    if all(q[x] <= ca[x] + cb[x] for x in range(3)):
                        H[:, :, ia * _nc(lb) + ib, h] = scale * cc * E[0].get((ca[0], cb[0], q[0]), zero) * E[1].get((ca[1], cb[1], q[1]), zero) * E[2].get((ca[2], cb[2], q[2]), zero)
        fa = torch.tensor([[off[a] + k for k in range(_nc(la))] for a, _ in pairs], device=dev)
        fb = torch.tensor([[off[b] + k for k in range(_nc(lb))] for _, b in pairs], device=dev)
        out.append(SimpleNamespace(L=la + lb, herm=herm, p=p, P=P, H=H, n=len(pairs), width=width, fa=fa[:, :, None].expand(-1, -1, fb.shape[1]).reshape(len(pairs), -1),
                                   fb=fb[:, None, :].expand(-1, fa.shape[1], -1).reshape(len(pairs), -1)))
    return out


def _exact_tensor(mol):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    n = mol.nbf
    G = torch.zeros((n, n, n, n), dtype=torch.float64, device=dev)
    cls = _exact_pairs(mol, dev)
    for x, bra in enumerate(cls):
        for ket in cls[:x + 1]:
            L = bra.L + ket.L
            q, Q = ket.p.reshape(-1), ket.P.reshape(-1, 3)
            sums = {tuple(np.add(t, u)) for t in bra.herm for u in ket.herm}
            step = max(1, int(2.5e8 / (len(_herm(L)) * 3 * bra.width * q.numel())))
            for s0 in range(0, bra.n, step):
                sl = slice(s0, min(bra.n, s0 + step))
                p, P = bra.p[sl].reshape(-1, 1), bra.P[sl].reshape(-1, 1, 3)
                d = P - Q
                alpha = p * q / (p + q)
                F = _boys(L, alpha * (d * d).sum(-1))
                pre = 2 * math.pi ** 2.5 / (p * q * torch.sqrt(p + q))
                R = {(0, 0, 0): [pre * (-2 * alpha) ** m * F[m] for m in range(L + 1)]}
                for tot in range(1, L + 1):  # R[t][m] for m <= L - |t|
                    for t in [h for h in _herm(L) if sum(h) == tot]:
                        ax = 0 if t[0] else 1 if t[1] else 2
                        t1 = tuple(v - (k == ax) for k, v in enumerate(t))
                        t2 = tuple(v - 2 * (k == ax) for k, v in enumerate(t))
                        R[t] = [d[..., ax] * R[t1][m + 1] + (t1[ax] * R[t2][m + 1] if t1[ax] else 0.0) for m in range(L - tot + 1)]
                R = {t: R[t][0] for t in sums}
                ns, na, nc = sl.stop - sl.start, bra.H.shape[2], ket.H.shape[2]
                Hb = bra.H[sl].permute(0, 2, 1, 3).reshape(ns, na, -1)
                block = torch.zeros((ns * na, ket.n, nc), dtype=torch.float64, device=dev)
                for iu, u in enumerate(ket.herm):
                    r = torch.stack([R[tuple(np.add(t, u))] for t in bra.herm], dim=1).reshape(ns, bra.width * len(bra.herm), -1)
                    w = torch.bmm(Hb, r).reshape(ns * na, ket.n, ket.width)
                    block += (-1) ** sum(u) * torch.einsum("akq,kqc->akc", w, ket.H[..., iu])
                block = block.reshape(ns, na, ket.n, nc)
                i, j = bra.fa[sl][:, :, None, None], bra.fb[sl][:, :, None, None]
                k, m = ket.fa[None, None], ket.fb[None, None]
                for a, b in ((i, j), (j, i)):
                    for c, e in ((k, m), (m, k)):
                        G[a, b, c, e] = block
                        G[c, e, a, b] = block
    return G


def exact(case, seed):
    kind = case["kind"]
    mol = _molecules(case, seed)[0]
    # a molecule whose tensor takes a few seconds; the gradient and the iterated kinds have no short 64-bit form
    if kind not in ("jk", "ujk", "stored", "mp2") or mol.nbf > 90 or int(mol.shell_l.max()) > 2:
        return None
    G = _exact_tensor(mol)
    n, dev = mol.nbf, G.device
    nocc = max(1, mol.n_electrons // 2)

    def jk(D, both=True):
        D = torch.tensor(D, device=dev) if not torch.is_tensor(D) else D
        return torch.einsum("ijkl,kl->ij", G, D), torch.einsum("ijkl,jk->il", G, D)

    if kind == "mp2":
        nocc = min(nocc, n - 1)
        C, e = torch.tensor(_orbitals(n, seed), device=dev), torch.tensor(_energies(n, nocc, seed), device=dev)
        v = torch.einsum("pqrs,pi,qa,rj,sb->iajb", G, C[:, :nocc], C[:, nocc:], C[:, :nocc], C[:, nocc:])
        den = e[:nocc, None, None, None] - e[None, nocc:, None, None] + e[None, None, :nocc, None] - e[None, None, None, nocc:]
        return float((v * (2 * v - v.permute(0, 3, 2, 1)) / den).sum())
    D = _density(n, nocc, seed, 0)
    if kind == "ujk":
        D2 = _density(n, max(1, nocc - 1), seed, 1)
        return jk(D + D2)[0], jk(D)[1], jk(D2)[1]
    J, K = jk(D)
    return (J, K) if kind == "jk" else (G, J, K)
