#!/usr/bin/env python3
"""Generate os_generated.cuh: straight-line 3c-CP integral code per shell-pair class.

The Obara-Saika vertical recursion (App. A, Eq. vrr) with early contraction.
With sigma = zeta_b / zeta, kappa = 1 / (2 zeta), AB = R_a - R_b and AC =
R_a - r_i, P - A = -sigma AB and P - r_i = AC - sigma AB, so that Eq. (vrr) reads

    Theta^n_{e+1_q} = - sigma AB_q (Theta^n_e - Theta^{n+1}_e) - AC_q Theta^{n+1}_e
                      + e_q kappa (Theta^n_{e-1_q} - Theta^{n+1}_{e-1_q}):

AB and AC do not depend on the primitive pair, sigma and kappa do not depend
on the point.  Unrolled down to the seeds S_n = pref F_n(T), every term is a
power sigma^i kappa^j of the primitive pair times the difference
W_{i+j,s} = sum_m (-1)^m C(i+j, m) S_{s+m} (i + 2j + s = |e|), times powers
of AB and AC.  The primitive pairs are therefore summed into the scalars

    M_{ijs} = sum_p sigma_p^i kappa_p^j W_{i+j,s}

first, and the recursion runs once per contracted pair on families
[e; i, j, s] with [0; i, j, s] = M_{ijs}:

    [e+1_q; i,j,s] = -AB_q [e; i+1,j,s] - AC_q [e; i,j,s+1] + e_q [e-1_q; i,j+1,s].

The W_{k,s} are integrals of t^{2s} (1 - t^2)^k e^{-T t^2} over [0, 1]: positive
and without cancellation, like the Boys functions themselves.

For each class (l_a, l_b) with l_a >= l_b, l <= 2 this emits

  * ``prim``: one primitive pair's differences, added into the NM scalars M;
  * ``build``: the recursion from M to [e; 0, 0, 0] for l_a <= |e| <= L, L = l_a + l_b;
  * ``hrr``: the horizontal recursion (App. A, Eq. hrr) to the target block Xi_{ab};
  * ``vrr``: the recursion for one primitive pair, as Eq. (vrr) states it: the FP32
    tier's pp, dp and dd, FP64 pairs of uncontracted shells, and the exports of a single
    shell pair's block;

as straight-line code on named registers, templated on the arithmetic type:
double (FP64 path), float (FP32 pairs of the mixed form) and ds (double-FP32).
Only what some target needs is emitted, and the directions of the recursion
steps are chosen (a seeded descent over all choices) for the fewest
operations.  The generator also counts the operations it emits (FMA = 2
flops), which the library reports as the algorithmic work of the integral
kernels.

Operations per primitive pair and per contracted pair (FMA counted once) with
this scheme, against the recursion run for every primitive pair:

    class       ss    ps      pp      ds      dp       dd
    primitive   1     3 / 9   9 / 37  7 / 34  16 / 88  29 / 180
    pair        0     6 / 0   42 / 9  27 / 0  118 / 22 313 / 79

Run:  python gen_os.py > os_generated.cuh
"""
from __future__ import annotations

import random
import sys

CLASSES = [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2)]


def ncart(l):
    return (l + 1) * (l + 2) // 2


def carts(l):
    return [(ax, ay, l - ax - ay) for ax in range(l, -1, -1) for ay in range(l - ax, -1, -1)]


def name_e(e):
    return f"{e[0]}{e[1]}{e[2]}"


def minus(e, q):
    return tuple(v - (i == q) for i, v in enumerate(e))


class Counter:
    def __init__(self):
        self.fma = self.mul = self.add = 0

    @property
    def flops(self):
        return 2 * self.fma + self.mul + self.add

    @property
    def ops(self):
        return self.fma + self.mul + self.add


def scalars(la, lb):
    """(i, j, s) of the contracted scalars: i + 2j + s = m for l_a <= m <= L."""
    return [(i, j, m - i - 2 * j) for m in range(la, la + lb + 1) for j in range(m // 2 + 1)
            for i in range(m - 2 * j + 1)]


def gen_prim(la, lb):
    """Seeds of one primitive pair into M; c(i, j) = sigma^i kappa^j are arguments (FP64: times the prefactor)."""
    L = la + lb
    ms = scalars(la, lb)
    need = set()

    def want(k, s):
        if (k, s) not in need:
            need.add((k, s))
            if k > 0:
                want(k - 1, s)
                want(k - 1, s + 1)

    for (i, j, s) in ms:
        want(i + j, s)
    c = Counter()
    lines = []
    for (k, s) in sorted(need):
        if k == 0:
            lines.append(f"const R w0_{s} = S[{s}];")
        else:
            lines.append(f"const R w{k}_{s} = w{k - 1}_{s} - w{k - 1}_{s + 1};")
            c.add += 1
    for n, (i, j, s) in enumerate(ms):
        if i == 0 and j == 0:
            lines.append(f"acc_lead(M[{n}], c.c00, w0_{s});")
            c.add += 1
        else:
            lines.append(f"acc_mac(M[{n}], c.c{i}{j}, w{i + j}_{s});")
            c.fma += 1
    return lines, c, {m: n for n, m in enumerate(ms)}


def gen_vrr(la, lb):
    """Eq. (vrr) of one primitive pair into the contracted accumulator acc."""
    targets = [(e, 0) for l in range(la, la + lb + 1) for e in carts(l)]

    def direction(e):  # the smallest positive component: no third term where it is 1
        return min((q for q in range(3) if e[q] > 0), key=lambda q: e[q])

    need = set()
    stack = list(targets)
    while stack:
        node = stack.pop()
        if node in need:
            continue
        need.add(node)
        e, n = node
        if sum(e) == 0:
            continue
        q = direction(e)
        m = minus(e, q)
        stack += [(m, n), (m, n + 1)]
        if m[q] > 0:
            stack += [(minus(m, q), n), (minus(m, q), n + 1)]
    c = Counter()
    lines = []
    for (e, n) in sorted(need, key=lambda x: (sum(x[0]), -x[0][0], -x[0][1], x[1])):
        v = f"t{name_e(e)}_{n}"
        if sum(e) == 0:
            lines.append(f"const R {v} = S[{n}];")
            continue
        q = direction(e)
        Q = "xyz"[q]
        m = minus(e, q)
        base = f"fma(PA{Q}, t{name_e(m)}_{n}, -PC{Q} * t{name_e(m)}_{n + 1})"
        c.fma += 1
        c.mul += 1
        if m[q] > 0:
            c.fma += 1
            c.add += 1
            mm = name_e(minus(m, q))
            base = f"fma(k{m[q]}, t{mm}_{n} - t{mm}_{n + 1}, {base})"
        lines.append(f"const R {v} = {base};")
    for k, (e, _) in enumerate(targets):
        lines.append(f"acc[{k}] += t{name_e(e)}_0;")
        c.add += 1
    return lines, c


def build_nodes(la, lb, dirs):
    need = set()
    stack = [(e, (0, 0, 0)) for l in range(la, la + lb + 1) for e in carts(l)]
    ops = 0
    while stack:
        node = stack.pop()
        if node in need:
            continue
        need.add(node)
        e, (i, j, s) = node
        if sum(e) == 0:
            continue
        q = dirs[e]
        m = minus(e, q)
        stack += [(m, (i + 1, j, s)), (m, (i, j, s + 1))]
        ops += 2
        if m[q] > 0:
            stack.append((minus(m, q), (i, j + 1, s)))
            ops += 1
    return need, ops


def choose_dirs(la, lb):
    es = [e for l in range(1, la + lb + 1) for e in carts(l)]
    best = None
    for seed in range(20):
        r = random.Random(seed)
        d = {e: r.choice([q for q in range(3) if e[q] > 0]) for e in es}
        n = build_nodes(la, lb, d)[1]
        for _ in range(400 if es else 0):
            e = r.choice(es)
            old = d[e]
            d[e] = r.choice([q for q in range(3) if e[q] > 0])
            m = build_nodes(la, lb, d)[1]
            if m <= n:
                n = m
            else:
                d[e] = old
        if best is None or n < best[0]:
            best = (n, dict(d))
    return best[1]


def gen_build(la, lb, m_index):
    """M -> acc[e] = [e; 0, 0, 0]; nAB = R_b - R_a, nAC = r_i - R_a."""
    dirs = choose_dirs(la, lb)
    need, _ = build_nodes(la, lb, dirs)
    c = Counter()
    lines = []

    def name(e, w):
        return f"v{name_e(e)}_{w[0]}{w[1]}{w[2]}"

    for (e, w) in sorted(need, key=lambda x: (sum(x[0]), -x[0][0], -x[0][1], x[1])):
        i, j, s = w
        if sum(e) == 0:
            lines.append(f"const R {name(e, w)} = acc_get(M[{m_index[w]}]);")
            continue
        q = dirs[e]
        Q = "xyz"[q]
        m = minus(e, q)
        args = f"nAB{Q}, {name(m, (i + 1, j, s))}, nAC{Q}, {name(m, (i, j, s + 1))}"
        c.mul += 1
        c.fma += 1
        if m[q] > 0:
            lines.append(f"const R {name(e, w)} = dot2_add<{m[q]}>({args}, {name(minus(m, q), (i, j + 1, s))});")
            if m[q] == 1:
                c.add += 1
            else:
                c.fma += 1
        else:
            lines.append(f"const R {name(e, w)} = dot2({args});")
    acc_index = {}
    for l in range(la, la + lb + 1):
        for e in carts(l):
            acc_index[e] = len(acc_index)
            lines.append(f"acc[{acc_index[e]}] = {name(e, (0, 0, 0))};")
    return lines, c, acc_index


def gen_hrr(la, lb, acc_index, rule):
    targets = [(a, b) for a in carts(la) for b in carts(lb)]
    need = set()
    stack = list(targets)

    def step(f):
        qs = [q for q in range(3) if f[q] > 0]
        return qs[0] if rule == 0 else qs[-1]

    while stack:
        node = stack.pop()
        if node in need:
            continue
        need.add(node)
        e, f = node
        if sum(f) == 0:
            continue
        q = step(f)
        g = minus(f, q)
        e1 = list(e)
        e1[q] += 1
        stack += [(tuple(e1), g), (e, g)]
    c = Counter()
    lines = []
    order = sorted(need, key=lambda x: (sum(x[1]), -sum(x[0]), x))
    for (e, f) in order:
        v = f"x{name_e(e)}_{name_e(f)}"
        if sum(f) == 0:
            lines.append(f"const R {v} = acc[{acc_index[e]}];")
            continue
        q = step(f)
        Q = "xyz"[q]
        g = minus(f, q)
        e1 = list(e)
        e1[q] += 1
        lines.append(f"const R {v} = fma(AB{Q}, x{name_e(e)}_{name_e(g)}, x{name_e(e1)}_{name_e(g)});")
        c.fma += 1
    for i, a in enumerate(carts(la)):
        for j, b in enumerate(carts(lb)):
            lines.append(f"xi[{i * ncart(lb) + j}] = x{name_e(a)}_{name_e(b)};")
    return lines, c


def main(out=sys.stdout):
    w = out.write
    w("// Generated by gen_os.py -- do not edit.\n")
    w("// Straight-line 3c-CP integral code of one shell-pair class: the Obara-Saika VRR\n")
    w("// (App. A, Eq. vrr) with the primitive pairs contracted into scalars first (the\n")
    w("// derivation is in gen_os.py), and the HRR (Eq. hrr), with the operation counts.\n")
    w("#pragma once\n\nnamespace snk {\n\n")
    w("// sigma^i kappa^j of one primitive pair, c<i><j>; a class reads those with i + 2j <= L.\n")
    w("// FP64: times the primitive pair's prefactor, c00 the prefactor itself; elsewhere the\n")
    w("// seeds carry the prefactor and c00 is not read (acc_lead)\n")
    w("template <typename R> struct OsCoef {\n  R c00, c10, c20, c30, c40, c01, c11, c21, c02;\n};\n\n")
    w("template <int LA, int LB> struct OsClass;\n\n")
    for (la, lb) in CLASSES:
        pl, pc, m_index = gen_prim(la, lb)
        bl, bc, acc_index = gen_build(la, lb, m_index)
        best = None
        for rule in (0, 1):
            hl, hc = gen_hrr(la, lb, acc_index, rule)
            if best is None or hc.ops < best[1].ops:
                best = (hl, hc)
        hl, hc = best
        vl, vc = gen_vrr(la, lb)
        L = la + lb
        w(f"// class ({la},{lb}): {pc.ops} operations ({pc.flops} flops) per primitive pair,\n")
        w(f"// {bc.ops + hc.ops} ({bc.flops + hc.flops} flops) per contracted pair\n")
        w(f"template <> struct OsClass<{la}, {lb}> {{\n")
        w(f"  static constexpr int L = {L};\n")
        w(f"  static constexpr int NM = {len(m_index)};\n")
        w(f"  static constexpr int NACC = {len(acc_index)};\n")
        w(f"  static constexpr int NA = {ncart(la)};\n")
        w(f"  static constexpr int NB = {ncart(lb)};\n")
        w(f"  static constexpr int PRIM_FLOPS = {pc.flops};\n")
        w(f"  static constexpr int PAIR_FLOPS = {bc.flops + hc.flops};\n")
        w(f"  static constexpr int VRR_FLOPS = {vc.flops};\n")
        w(f"  static constexpr int HRR_FLOPS = {hc.flops};\n")
        w("  template <typename R, typename A>\n")
        w("  __device__ static __forceinline__ void prim(const R* S, const OsCoef<R>& c, A* M) {\n")
        w("    (void)c;\n")
        for s in pl:
            w("    " + s + "\n")
        w("  }\n")
        w("  template <typename R, typename A>\n")
        w("  __device__ static __forceinline__ void build(const A* M, R nABx, R nABy, R nABz, R nACx, R nACy, R nACz,\n")
        w("                                               R* acc) {\n")
        w("    (void)nABx; (void)nABy; (void)nABz; (void)nACx; (void)nACy; (void)nACz;\n")
        for s in bl:
            w("    " + s + "\n")
        w("  }\n")
        w("  template <typename R, typename A>\n")
        w("  __device__ static __forceinline__ void vrr(const R* S, R PAx, R PAy, R PAz, R PCx, R PCy, R PCz,\n")
        w("                                             R k1, R k2, R k3, A* acc) {\n")
        w("    (void)PAx; (void)PAy; (void)PAz; (void)PCx; (void)PCy; (void)PCz; (void)k1; (void)k2; (void)k3;\n")
        for s in vl:
            w("    " + s + "\n")
        w("  }\n")
        w("  template <typename R>\n")
        w("  __device__ static __forceinline__ void hrr(const R* acc, R ABx, R ABy, R ABz, R* xi) {\n")
        w("    (void)ABx; (void)ABy; (void)ABz;\n")
        for s in hl:
            w("    " + s + "\n")
        w("  }\n};\n\n")
    w("}  // namespace snk\n")


if __name__ == "__main__":
    main()
