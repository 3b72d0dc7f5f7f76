"""The work that users of the library have it do, as cases that can be timed and compared.

Each case goes through the package's public entry points on inputs made from a
seed: a globular cluster of O- and H-like atoms (one in three heavy, 0.08 atoms
per cubic Angstrom), even-tempered contracted Cartesian shells up to d, an
atom-centred product grid with Becke weights and a localised projector density,
the recipes of the repository's own workloads.  What is kept in the state is
what a self-consistent-field program keeps: the handle of the geometry, the
density on the device and the output buffer.  A pass is one density: load it
(which runs the density-dependent screen) and build.

`exact` evaluates the same quantities in 64 bits with plain torch: unscreened
exchange by Obara-Saika recursions on Boys functions interpolated from torch's
incomplete gamma function, the exchange-correlation potential with automatic
differentiation of the energy density, and the gradient of the screen network
by automatic differentiation.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2303_14280_gb300 as snk

BOHR = 1.0 / 0.529177210903
# shells (l, j) per element; shell j has the exponents 0.1 * 3^(3j..3j+2)
RECIPES = {"small": {8: [(0, 0), (0, 1), (0, 2), (1, 0), (1, 1), (2, 0)], 1: [(0, 0), (0, 1)]},
           "scale": {8: [(0, 0), (0, 1), (0, 2), (1, 0), (1, 1), (2, 0), (2, 1)], 1: [(0, 0), (0, 1), (1, 0)]}}
# the forms of the library a user picks from
FORMS = {
    "plain": dict(),
    "double_fp32": dict(precision="mixed", fp32_bound=0.0, ds_integrals=1, gemm="df32"),
    "mixed": dict(eps=1e-10, precision="mixed", fp32_bound=3e-4, ds_integrals=1, gemm="split", tc_slices_hi=5,
                  tc_slices_lo=4, eps_tile=1e-11),
}
GRIDS = [(16, 4, 9), (20, 5, 10), (40, 5, 15), (40, 8, 15), (50, 8, 15), (50, 8, 20)]
FUNCTIONALS = {"lda_x": 1, "pbe_x": 2, "pbe": 3}


def listed():
    return [
        # one small molecule in the default FP64 form: launches, copies and waits count
        dict(name="chain4_plain", what="K", form="plain", atoms=4, recipe="small", n_r=40, n_th=5, n_ph=15),
        # an ordinary molecule in the default form
        dict(name="mol24_plain", what="K", form="plain", atoms=24, recipe="scale", n_r=40, n_th=5, n_ph=15),
        # the FP64-grade form on the FP32 pipe, ragged batches
        dict(name="mol17_double_fp32", what="K", form="double_fp32", atoms=17, recipe="scale", n_r=50, n_th=8, n_ph=15),
        # a single point on a coarse grid, the mixed form without trained weights
        dict(name="mol12_mixed", what="K", form="mixed", atoms=12, recipe="scale", n_r=40, n_th=8, n_ph=15),
        # an ordinary molecule in the mixed form with the shipped screen weights
        dict(name="mol32_learned", what="K", form="mixed", learned=True, atoms=32, recipe="scale", n_r=50, n_th=8,
             n_ph=20),
        # the 96-atom cluster of the benchmark in the mixed form with the screen weights
        dict(name="mol96_learned", what="K", form="mixed", learned=True, atoms=96, recipe="scale", n_r=50, n_th=8,
             n_ph=20),
        # alpha and beta densities of an open shell in one build, host arrays in and out
        dict(name="mol16_two_densities", what="K2", form="mixed", atoms=16, recipe="scale", n_r=40, n_th=8, n_ph=15),
        # many small molecules in one handle, replayed from a graph
        dict(name="batch24_double_fp32", what="batch", form="double_fp32", molecules=24, recipe="scale", n_r=40, n_th=5,
             n_ph=15),
        # the semilocal half of a hybrid functional: PBE potential, FP64 tiles
        dict(name="mol20_vxc_plain", what="vxc", form="plain", fun="pbe", atoms=20, recipe="scale", n_r=40, n_th=8,
             n_ph=15),
        # the same for the 96-atom cluster with tensor-core products
        dict(name="mol96_vxc_mixed", what="vxc", form="mixed", fun="pbe", atoms=96, recipe="scale", n_r=50, n_th=8,
             n_ph=20),
        # one gradient step's worth of training blocks of the learned screen
        dict(name="screen_grad", what="grad", rows=32768),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["plain", "double_fp32", "mixed", "mixed", "learned", "learned", "K2", "batch", "vxc", "vxc",
                       "grad"])
    if what == "grad":
        return dict(what="grad", rows=_logint(rng, 513, 40000))
    n_r, n_th, n_ph = rng.choice(GRIDS)
    g = dict(n_r=n_r, n_th=n_th, n_ph=n_ph)
    if what == "plain":
        return dict(what="K", form="plain", atoms=_logint(rng, 3, 18), recipe=rng.choice(["small", "scale"]), **g)
    if what == "double_fp32":
        return dict(what="K", form="double_fp32", atoms=_logint(rng, 4, 24), recipe="scale", **g)
    if what == "mixed":
        return dict(what="K", form="mixed", atoms=_logint(rng, 6, 48), recipe="scale", **g)
    if what == "learned":
        return dict(what="K", form="mixed", learned=True, atoms=_logint(rng, 12, 80), recipe="scale", **g)
    if what == "K2":
        return dict(what="K2", form=rng.choice(["plain", "mixed"]), atoms=_logint(rng, 4, 14), recipe="scale", **g)
    if what == "batch":
        return dict(what="batch", form=rng.choice(["plain", "double_fp32"]), molecules=_logint(rng, 3, 24),
                    recipe="scale", n_r=rng.choice([16, 20, 40]), n_th=5, n_ph=rng.choice([10, 15]))
    form = rng.choice(["plain", "double_fp32", "mixed", "mixed"])
    return dict(what="vxc", form=form, fun=rng.choice(sorted(FUNCTIONALS)),
                atoms=_logint(rng, 3, 80 if form == "mixed" else 20), recipe=rng.choice(["small", "scale"]), **g)


# ------------------------------------------------------------------ inputs

def _geometry(n_atoms, rng):
    """Random sequential placement in a sphere, pairs at least 1 Angstrom apart; one atom in three heavy."""
    radius = (3.0 * n_atoms / 0.08 / (4.0 * math.pi)) ** (1.0 / 3.0)
    pos = np.zeros((0, 3))
    while pos.shape[0] < n_atoms:
        p = rng.uniform(-radius, radius, size=3)
        if p @ p <= radius * radius and (not len(pos) or np.min(np.sum((pos - p) ** 2, axis=1)) >= 1.0):
            pos = np.vstack([pos, p])
    Z = np.ones(n_atoms, dtype=np.int32)
    Z[rng.permutation(n_atoms)[:max(1, n_atoms // 3)]] = 8
    return Z, pos * BOHR


def _basis(Z, xyz, recipe, rng):
    l, atom, center, exps, coefs = [], [], [], [], []
    for a, z in enumerate(Z):
        for (la, j) in RECIPES[recipe][int(z)]:
            l.append(la)
            atom.append(a)
            center.append(xyz[a])
            exps += [0.1 * 3.0 ** (3 * j + k) for k in range(3)]
            coefs += list(1.0 - 0.8 * rng.random(3))
    return SimpleNamespace(l=np.array(l, dtype=np.int32), nprim=np.full(len(l), 3, dtype=np.int32),
                           atom=np.array(atom, dtype=np.int32), center=np.array(center), exps=np.array(exps),
                           coefs=np.array(coefs))


def _n_functions(basis):
    return int(sum((int(l) + 1) * (int(l) + 2) // 2 for l in basis.l))


def _grid(xyz, n_r, n_th, n_ph):
    """Mura-Knowles radial (alpha 5) x Gauss-Legendre x trapezoid around every atom, Becke partition weights."""
    x = (np.arange(1, n_r + 1) - 0.5) / n_r
    r = -5.0 * np.log1p(-x ** 3)
    wr = r * r * 15.0 * x ** 2 / ((1.0 - x ** 3) * n_r)
    ct, wt = np.polynomial.legendre.leggauss(n_th)
    phi = 2.0 * math.pi * (np.arange(n_ph) + 0.5) / n_ph
    st = np.sqrt(1.0 - ct ** 2)
    dirs = np.stack([np.outer(st, np.cos(phi)), np.outer(st, np.sin(phi)), np.outer(ct, np.ones(n_ph))], axis=-1)
    rel = (r[:, None, None] * dirs.reshape(-1, 3)[None]).reshape(-1, 3)
    w1 = (wr[:, None] * np.outer(wt, np.full(n_ph, 2.0 * math.pi / n_ph)).reshape(-1)[None]).reshape(-1)
    n_at, n_pt = xyz.shape[0], rel.shape[0]
    pts = (xyz[:, None, :] + rel[None]).reshape(-1, 3)
    owner = np.repeat(np.arange(n_at, dtype=np.int32), n_pt)
    w = np.tile(w1, n_at)
    if n_at > 1:
        A = torch.as_tensor(xyz, device="cuda")
        R = torch.cdist(A, A)
        inv = torch.where(R > 0, 1.0 / torch.where(R > 0, R, 1.0), 0.0)
        eye = torch.eye(n_at, dtype=torch.bool, device="cuda")
        part = torch.empty(len(w), dtype=torch.float64, device="cuda")
        dp, own = torch.as_tensor(pts, device="cuda"), torch.as_tensor(owner, device="cuda").long()
        step = max(256, (1 << 25) // (n_at * n_at))
        for s in range(0, len(w), step):
            d = (dp[s:s + step, None, :] - A[None]).square().sum(-1).sqrt()
            f = (d[:, :, None] - d[:, None, :]) * inv
            for _ in range(3):
                f = f * (1.5 - 0.5 * f * f)
            f = (0.5 - 0.5 * f).masked_fill_(eye, 1.0).prod(dim=2)
            part[s:s + step] = f.gather(1, own[s:s + step, None])[:, 0] / f.sum(1)
        w = w * part.cpu().numpy()
    return SimpleNamespace(xyz=np.ascontiguousarray(pts), w=w, atom=owner)


def _density(xyz, basis, n_occ, rng):
    """Projector on n_occ random orbitals with Gaussian envelopes (3 bohr) around random atoms."""
    nf = np.array([(int(l) + 1) * (int(l) + 2) // 2 for l in basis.l])
    fc = np.repeat(basis.center, nf, axis=0)
    C = rng.normal(size=(fc.shape[0], n_occ))
    d2 = ((fc[:, None, :] - xyz[rng.integers(0, xyz.shape[0], size=n_occ)][None]) ** 2).sum(-1)
    C *= np.exp(-d2 / 18.0)
    ev, U = np.linalg.eigh(C.T @ C)
    C = C @ (U / np.sqrt(ev)) @ U.T
    P = C @ C.T
    return 0.5 * (P + P.T)


def _molecule(case, seed, atoms=None, n_dens=1):
    rng = np.random.default_rng(seed)
    Z, xyz = _geometry(atoms or case["atoms"], rng)
    basis = _basis(Z, xyz, case["recipe"], rng)
    n_occ = int(math.ceil(0.2 * _n_functions(basis)))
    P = [_density(xyz, basis, max(1, n_occ - d), rng) for d in range(n_dens)]
    return basis, _grid(xyz, case["n_r"], case["n_th"], case["n_ph"]), P


def _batch(case, seed):
    sizes = np.random.default_rng(7919 + case["molecules"]).integers(4, 13, size=case["molecules"])
    return [_molecule(case, seed * 1000 + m, atoms=int(n)) for m, n in enumerate(sizes)]


def _screen_rows(case, seed):
    """Feature rows and labels spread like the screen's own, and the shipped weights."""
    g = torch.Generator().manual_seed(seed)
    X = torch.randn(case["rows"], snk.MLP_FEATURES, generator=g) * 0.5
    Y = -1.0 + 0.3 * torch.randn(case["rows"], generator=g)
    w = torch.as_tensor(snk.trained_screen()[0]) * (1.0 + 0.05 * torch.randn(snk.MLP_WEIGHTS, generator=g))
    return w.numpy(), X.numpy(), Y.numpy()


def prepare(case, seed):
    what = case["what"]
    if what == "grad":
        w, X, Y = _screen_rows(case, seed)
        return SimpleNamespace(what=what, w=w, X=X, Y=Y)
    opts = dict(FORMS[case["form"]])
    if what == "batch":
        mols = _batch(case, seed)
        eng = snk.Engine([m[0] for m in mols], [m[1] for m in mols], graph=1, **opts)
        P = torch.as_tensor(np.concatenate([m[2][0].reshape(-1) for m in mols]), device="cuda")
        return SimpleNamespace(what="K", eng=eng, P=P, out=torch.empty_like(P))
    basis, grid, P = _molecule(case, seed, n_dens=2 if what == "K2" else 1)
    if case.get("learned"):
        w, skip, meta = snk.trained_screen()
        opts.update(screen="learned", learned_skip=skip, learned_fp32=meta["fp32_threshold"])
    eng = snk.Engine(basis, grid, **opts)
    if case.get("learned"):
        eng.screen_load(w)
    if what == "K2":
        return SimpleNamespace(what=what, eng=eng, P=P)
    dP = torch.as_tensor(P[0], device="cuda")
    s = SimpleNamespace(what=what, eng=eng, P=dP, out=torch.empty_like(dP))
    if what == "vxc":
        s.fun = FUNCTIONALS[case["fun"]]
        eng.set_density(dP)
    return s


def run(s):
    if s.what == "grad":
        return snk.mlp_grad(s.w, s.X, s.Y)
    if s.what == "vxc":
        return s.eng.build_Vxc(s.fun, out=s.out)
    s.eng.set_density(s.P)
    return s.eng.build_K() if s.what == "K2" else s.eng.build_K(out=s.out)


# ------------------------------------------------------------------ work

def _counts(atoms, case):
    """(points, functions, shells, work of one point's integrals) of a molecule: per shell pair the contraction
    with F in both directions and, per primitive pair, a distance and one Boys function."""
    rec = RECIPES[case["recipe"]]
    heavy = max(1, atoms // 3)
    shells = heavy * [l for l, _ in rec[8]] + (atoms - heavy) * [l for l, _ in rec[1]]
    nf = sum((l + 1) * (l + 2) // 2 for l in shells)
    return atoms * case["n_r"] * case["n_th"] * case["n_ph"], nf, len(shells), 2.0 * nf * nf + \
        0.5 * len(shells) * (len(shells) + 1) * 9 * 20.0


def work(case):
    if case["what"] == "grad":
        n = case["rows"]
        return {"bytes": 4.0 * (17 * n + 2 * snk.MLP_WEIGHTS), "flops": 6.0 * n * (16 * 64 + 2 * 64 * 64 + 64)}
    sizes = [case["atoms"]] if case["what"] != "batch" else \
        [int(n) for n in np.random.default_rng(7919 + case["molecules"]).integers(4, 13, size=case["molecules"])]
    nd = 2 if case["what"] == "K2" else 1
    b = f = 0.0
    for n in sizes:
        pts, nf, ns, ints = _counts(n, case)
        b += 32.0 * pts + 16.0 * nd * nf * nf
        f += pts * nf * nf * 4.0 * nd + (0.0 if case["what"] == "vxc" else pts * ints)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64-bit values

def _carts(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _dfact(n):
    return 1.0 if n <= 0 else n * _dfact(n - 2)


class _Shells:
    """Normalised shells of a basis: unit self-overlap of every Cartesian component."""

    def __init__(self, basis):
        self.l = [int(v) for v in basis.l]
        self.c = np.asarray(basis.center)
        self.a = np.asarray(basis.exps).reshape(-1, 3)
        d = np.asarray(basis.coefs).reshape(-1, 3).copy()
        self.first = np.concatenate([[0], np.cumsum([(l + 1) * (l + 2) // 2 for l in self.l])]).astype(int)
        self.nf = int(self.first[-1])
        self.f = np.ones(self.nf)
        for s, l in enumerate(self.l):
            a = self.a[s]
            d[s] *= (2 * a / math.pi) ** 0.75 * (4 * a) ** (l / 2) / math.sqrt(_dfact(2 * l - 1))
            g = a[:, None] + a[None, :]
            d[s] /= math.sqrt(np.sum(d[s][:, None] * d[s][None, :] * (math.pi / g) ** 1.5 * _dfact(2 * l - 1) / (2 * g) ** l))
            for k, e in enumerate(_carts(l)):
                self.f[self.first[s] + k] = math.sqrt(_dfact(2 * l - 1) / np.prod([_dfact(2 * q - 1) for q in e]))
        self.d = d

    def phi(self, r, grad=False):
        """Functions (and their three derivatives) at the points r (n, 3): (nf, n) each."""
        out = torch.empty((4 if grad else 1, self.nf, r.shape[0]), dtype=torch.float64, device=r.device)
        for s, l in enumerate(self.l):
            x = r - torch.as_tensor(self.c[s], device=r.device)
            r2 = x.square().sum(1)
            e = [float(self.d[s, k]) * torch.exp(-float(self.a[s, k]) * r2) for k in range(3)]
            R0 = e[0] + e[1] + e[2]
            R1 = sum(-2.0 * float(self.a[s, k]) * e[k] for k in range(3)) if grad else None
            p = [[x[:, q] ** n if n >= 0 else None for n in range(l + 1)] for q in range(3)]
            for k, c in enumerate(_carts(l)):
                i = self.first[s] + k
                m = p[0][c[0]] * p[1][c[1]] * p[2][c[2]]
                out[0, i] = self.f[i] * m * R0
                for q in range(3 if grad else 0):
                    o = p[(q + 1) % 3][c[(q + 1) % 3]] * p[(q + 2) % 3][c[(q + 2) % 3]]
                    dm = c[q] * p[q][c[q] - 1] * o * R0 if c[q] else 0.0
                    out[1 + q, i] = self.f[i] * (dm + m * x[:, q] * R1)
        return out


_BOYS = {}


def _boys(L, T):
    """F_0..F_L(T): F_L by Taylor steps from nodes 1/16 apart (F_n' = -F_{n+1}), then downward recursion."""
    if "table" not in _BOYS:
        t = torch.arange(0, 16 * 46 + 2, dtype=torch.float64, device="cuda") / 16.0
        rows = []
        for n in range(16):
            a = torch.full_like(t, n + 0.5)
            small = torch.stack([(-t) ** k / (float(math.factorial(k)) * (2 * n + 2 * k + 1)) for k in range(40)]).sum(0)
            v = torch.special.gammainc(a, t.clamp_min(1e-3)) * math.gamma(n + 0.5) / (2.0 * t.clamp_min(1e-3) ** (n + 0.5))
            rows.append(torch.where(t < 1.0, small, v))
        _BOYS["table"] = torch.stack(rows)
    tab = _BOYS["table"]
    near = T < 46.0
    Tn = torch.where(near, T, 1.0)
    k = torch.round(Tn * 16.0).long()
    x = k.double() / 16.0 - Tn
    f = tab[L + 10][k] / math.factorial(10)
    for m in range(9, -1, -1):
        f = f * x + tab[L + m][k] / math.factorial(m)
    F = [None] * (L + 1)
    F[L] = f
    e = torch.exp(-Tn) if L else None
    for n in range(L - 1, -1, -1):
        F[n] = (2.0 * Tn * F[n + 1] + e) / (2 * n + 1)
    Tf = torch.where(near, 1.0, T)
    g = 0.5 * torch.sqrt(math.pi / Tf)
    for n in range(L + 1):
        F[n] = torch.where(near, F[n], g)
        g = g * (2 * n + 1) / (2.0 * Tf)
    return F


def _class_blocks(la, lb, zeta, PA, AB, pref, r_minus, n_pairs):
    """Contracted blocks {(a, b): (pairs, points)} of one class; zeta, pref (prims, 1), PA, r_minus = P - r."""
    L = la + lb
    T = zeta * (r_minus[0] ** 2 + r_minus[1] ** 2 + r_minus[2] ** 2)
    F = _boys(L, T)
    memo = {((0, 0, 0), n): pref * F[n] for n in range(L + 1)}
    k = 0.5 / zeta

    def theta(e, n):
        if (e, n) not in memo:
            q = min((i for i in range(3) if e[i] > 0), key=lambda i: e[i])
            m = tuple(e[i] - (i == q) for i in range(3))
            v = PA[q] * theta(m, n) - r_minus[q] * theta(m, n + 1)
            if m[q]:
                mm = tuple(m[i] - (i == q) for i in range(3))
                v = v + (m[q] * k) * (theta(mm, n) - theta(mm, n + 1))
            memo[(e, n)] = v
        return memo[(e, n)]

    acc = {(e, (0, 0, 0)): theta(e, 0).view(n_pairs, 9, -1).sum(1) for l in range(la, L + 1) for e in _carts(l)}

    def hrr(e, f):
        if (e, f) not in acc:
            q = next(i for i in range(3) if f[i] > 0)
            g = tuple(f[i] - (i == q) for i in range(3))
            acc[(e, f)] = hrr(tuple(e[i] + (i == q) for i in range(3)), g) + AB[q] * hrr(e, g)
        return acc[(e, f)]

    return [[hrr(a, b) for b in _carts(lb)] for a in _carts(la)]


def _exact_K(basis, grid, Ps):
    """K of every density, unscreened (pairs whose charge overlaps below 1e-19 are left out)."""
    sh = _Shells(basis)
    dev = torch.device("cuda")
    r, w = torch.as_tensor(grid.xyz, device=dev), torch.as_tensor(grid.w, device=dev)
    P = [torch.as_tensor(p, device=dev) for p in Ps]
    f = torch.as_tensor(sh.f, device=dev)
    phi = sh.phi(r)[0]
    F = [p @ phi for p in P]
    G = [torch.zeros_like(phi) for _ in P]
    by = {}
    for a in range(len(sh.l)):
        for b in range(len(sh.l)):
            if sh.l[a] > sh.l[b] or (sh.l[a] == sh.l[b] and a >= b):
                amin = sh.a[a].min() * sh.a[b].min() / (sh.a[a].min() + sh.a[b].min())
                if amin * np.sum((sh.c[a] - sh.c[b]) ** 2) < 60.0:
                    by.setdefault((sh.l[a], sh.l[b]), []).append((a, b))
    n_pt = r.shape[0]
    for (la, lb), pairs in by.items():
        group = max(1, int(1.2e7 // (9 * n_pt)))
        pt_step = n_pt if group > 1 else max(1, int(1.2e7 // 9))
        for g0 in range(0, len(pairs), group):
            pg = np.array(pairs[g0:g0 + group])
            A, B = sh.c[pg[:, 0]], sh.c[pg[:, 1]]
            al, be = np.repeat(sh.a[pg[:, 0]], 3, axis=1), np.tile(sh.a[pg[:, 1]], (1, 3))
            z = al + be
            Pc = (al[..., None] * A[:, None] + be[..., None] * B[:, None]) / z[..., None]
            dd = np.repeat(sh.d[pg[:, 0]], 3, axis=1) * np.tile(sh.d[pg[:, 1]], (1, 3))
            pref = 2 * math.pi / z * np.exp(-al * be / z * np.sum((A - B) ** 2, axis=1)[:, None]) * dd

            def t(v):
                return torch.as_tensor(np.ascontiguousarray(v), device=dev).reshape(-1, 1)
            PA = [t(Pc[..., q] - A[:, None, q]) for q in range(3)]
            AB = [t(A[:, q] - B[:, q]) for q in range(3)]
            ia = torch.as_tensor(sh.first[pg[:, 0]], device=dev)
            ib = torch.as_tensor(sh.first[pg[:, 1]], device=dev)
            off = torch.as_tensor((pg[:, 0] != pg[:, 1]).astype(float), device=dev)[:, None]
            for p0 in range(0, n_pt, pt_step):
                sl = slice(p0, p0 + pt_step)
                rm = [t(Pc[..., q]) - r[None, sl, q] for q in range(3)]
                blk = _class_blocks(la, lb, t(z), PA, AB, t(pref), rm, len(pg))
                for u in range(len(blk)):
                    for v in range(len(blk[0])):
                        x = blk[u][v] * (f[ia + u] * f[ib + v])[:, None]
                        for d in range(len(P)):
                            G[d][:, sl].index_add_(0, ia + u, x * F[d][ib + v, sl])
                            G[d][:, sl].index_add_(0, ib + v, off * x * F[d][ia + u, sl])
    out = []
    for d in range(len(P)):
        K = (G[d] * w) @ phi.T
        out.append(0.5 * (K + K.T))
    return out


def _energy_density(fun, rho, gamma):
    """eps(rho, gamma) of Slater exchange, PBE exchange or PBE."""
    ex = -0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * rho ** (4.0 / 3.0)
    if fun == 1:
        return ex + 0.0 * gamma
    kappa, beta = 0.804, 0.06672455060314922
    mu = beta * math.pi ** 2 / 3.0
    kf = (3.0 * math.pi ** 2 * rho) ** (1.0 / 3.0)
    s2 = gamma / (4.0 * kf ** 2 * rho ** 2)
    e = ex * (1.0 + kappa - kappa / (1.0 + mu * s2 / kappa))
    if fun == 2:
        return e
    a, a1, b = 0.031091, 0.21370, (7.5957, 3.5876, 1.6382, 0.49294)
    rs = (3.0 / (4.0 * math.pi * rho)) ** (1.0 / 3.0)
    q = rs.sqrt()
    ec = -2.0 * a * (1.0 + a1 * rs) * torch.log1p(1.0 / (2.0 * a * q * (b[0] + q * (b[1] + q * (b[2] + q * b[3])))))
    g = (1.0 - math.log(2.0)) / math.pi ** 2
    t2 = math.pi * gamma / (16.0 * kf * rho ** 2)
    A = (beta / g) / torch.expm1(-ec / g)
    z = A * t2
    return e + rho * (ec + g * torch.log1p((beta / g) * t2 * (1.0 + z) / (1.0 + z + z * z)))


def _exact_vxc(basis, grid, P, fun):
    sh = _Shells(basis)
    P = torch.as_tensor(P, device="cuda")
    V = torch.zeros_like(P)
    E = 0.0
    step = max(1024, int(1.5e9 // (32 * sh.nf)))
    for s in range(0, len(grid.w), step):
        r = torch.as_tensor(grid.xyz[s:s + step], device="cuda")
        w = torch.as_tensor(grid.w[s:s + step], device="cuda")
        phi = sh.phi(r, grad=True)
        F = P @ phi[0]
        rho = (F * phi[0]).sum(0)
        g = [2.0 * (F * phi[1 + q]).sum(0) for q in range(3)]
        keep = rho >= 1e-14
        rk = torch.where(keep, rho, 1.0).requires_grad_(True)
        gk = torch.where(keep, g[0] ** 2 + g[1] ** 2 + g[2] ** 2, 0.0).requires_grad_(True)
        eps = _energy_density(fun, rk, gk)
        vr, vg = torch.autograd.grad(eps.sum(), (rk, gk))
        E += float((w * torch.where(keep, eps.detach(), 0.0)).sum())
        vr, vg = torch.where(keep, vr, 0.0), torch.where(keep, vg, 0.0)
        Z = 0.5 * w * (vr * phi[0] + 4.0 * vg * (g[0] * phi[1] + g[1] * phi[2] + g[2] * phi[3]))
        V += phi[0] @ Z.T
    return V + V.T, E


def _exact_grad(w, X, Y, under=4.0):
    w = torch.as_tensor(w).double().cuda().requires_grad_(True)
    X, Y = torch.as_tensor(X).double().cuda(), torch.as_tensor(Y).double().cuda()
    o = 0
    h = X
    for n_in, n_out in ((16, 64), (64, 64), (64, 64), (64, 1)):
        W, b = w[o:o + n_in * n_out].view(n_in, n_out), w[o + n_in * n_out:o + n_in * n_out + n_out]
        o += n_in * n_out + n_out
        h = h @ W + b
        if n_out > 1:
            h = torch.relu(h)
    r = h[:, 0] - Y
    loss = (torch.where(r < 0, under, 1.0) * r * r).mean()
    loss.backward()
    return float(loss), w.grad


def exact(case, seed):
    what = case["what"]
    if what == "grad":
        return _exact_grad(*_screen_rows(case, seed))
    if what == "batch":
        pts = sum(_counts(len(set(m[0].atom)), case)[0] * len(m[0].l) ** 2 for m in _batch(case, seed))
        if pts > 8e8:
            return None
        return torch.cat([_exact_K(b, g, P)[0].reshape(-1) for b, g, P in _batch(case, seed)])
    pts, nf, ns, _ = _counts(case["atoms"], case)
    if what == "vxc":
        if pts * float(nf) ** 2 > 1.2e12:
            return None
        basis, grid, P = _molecule(case, seed)
        return _exact_vxc(basis, grid, P[0], FUNCTIONALS[case["fun"]])
    if pts * float(ns) ** 2 > 8e8:
        return None
    basis, grid, P = _molecule(case, seed, n_dens=2 if what == "K2" else 1)
    K = _exact_K(basis, grid, P)
    return K if what == "K2" else K[0]
