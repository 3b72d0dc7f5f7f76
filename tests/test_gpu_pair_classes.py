"""The builds' contracted integral code, one shell-pair class at a time.

A two-shell molecule on a few points (both centres, the midpoint, near and far)
makes K the contraction of that class's blocks (and of the two diagonal ones),
for every class, for one to sixteen primitives per shell, and for point counts
around the 64- and 128-point tiles.

Tolerance: a block is a chain of at most 64 roundings (Boys seeds, contraction,
recursion) of terms no larger than the pair's rigorous bound times
(1 + |AB|^2)^2 for the powers of AB that cancel in the horizontal recursion, so
|dK| <= 64 u (1 + |AB|^2)^2 sum_i w_i |F|_max |Phi|_max bound, with u = 2^-53
(FP64), 2^-46 (double-FP32: one operation's error) and 2^-21 (FP32 tier: the
hardware exponential).  Ten times the FP64 value leaves room for the oracle's
own rounding.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

FORMS = {
    "fp64": (dict(screen="none"), 640 * 2.0 ** -53),
    "ds": (dict(screen="none", precision="mixed", fp32_bound=0.0, ds_integrals=1), 64 * 2.0 ** -46),
    "fp32": (dict(eps_E=0.0, eps_K=0.0, precision="mixed", fp32_bound=1e30), 64 * 2.0 ** -21),
}


def _case(la, lb, na, nb, apart, n_points, seed):
    rng = np.random.default_rng(seed)
    A = np.array([0.3, -0.7, 1.1])
    B = A + (np.array([1.1, 0.6, -0.9]) if apart else 0.0)
    basis = synth.Basis(l=np.array([la, lb], dtype=np.int32), nprim=np.array([na, nb], dtype=np.int32),
                        atom=np.array([0, 1], dtype=np.int32), center=np.stack([A, B]),
                        exps=np.exp(rng.uniform(np.log(0.15), np.log(30.0), na + nb)),
                        coefs=rng.uniform(0.2, 1.0, na + nb))
    pts = np.concatenate([A[None], B[None], 0.5 * (A + B)[None], A + rng.normal(size=(n_points, 3)) * 0.8,
                          A + rng.normal(size=(n_points, 3)) * 5.0])[:n_points]
    grid = synth.Grid(xyz=np.ascontiguousarray(pts), w=rng.uniform(0.5, 1.5, n_points),
                      atom=np.zeros(n_points, dtype=np.int32))
    P = rng.normal(size=(basis.n_functions,) * 2)
    return basis, grid, 0.5 * (P + P.T)


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("la,lb", [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (0, 2), (1, 2)])
def test_two_shell_exchange_matches_oracle(form, la, lb):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    opts, u = FORMS[form]
    for k, (na, nb, apart, n) in enumerate([(1, 1, True, 1), (3, 3, True, 127), (3, 2, False, 129), (16, 1, True, 64),
                                            (16, 16, True, 65), (5, 4, True, 300)]):
        basis, grid, P = _case(la, lb, na, nb, apart, n, 100 * la + 10 * lb + k)
        eng = snk.Engine(basis, grid, eps_basis=0.0, **opts)
        eng.set_density(P)
        K = eng.build_K()
        bound = max(eng.debug_pair_bound(a, b) for a in (0, 1) for b in (0, 1))
        st = eng.stats()
        eng.close()
        assert (st["pairs_kept_fp32"] > 0) == (form == "fp32")
        Phi = oracle.collocation(basis, grid.xyz).T
        F = P @ Phi
        ab2 = float(np.sum((basis.center[0] - basis.center[1]) ** 2))
        tol = u * (1.0 + ab2) ** 2 * bound * float(np.sum(grid.w * np.abs(F).sum(0) * np.abs(Phi).max(0)))
        err = np.max(np.abs(K - oracle.snk_K(basis, grid, P)))
        assert err <= tol, f"{form} l=({la},{lb}) primitives ({na},{nb}) points {n}: {err:.3e} > {tol:.3e}"
