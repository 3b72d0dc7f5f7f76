"""Products and collocation at the edges of their tiles.

Molecules of n s and p shells on a few points put the FP64 and double-FP32
products at 1, 16, 17, 64, 65 and more functions and at point counts where the
blocks share the points (one block's 64 points, remainders, one point), and
the collocation's exponentials over alpha r^2 from 0 to beyond the cut at 60
(exponents from 1e-3 to 1e4, points on centres and far away).

Tolerance: every entry is a sum of products of a few rounded factors; 512
units of 2^-53 (FP64) or 2^-46 (double-FP32) of the sum of the products'
absolute values covers the roundings of the factors (the exponential and the
powers about 8 each, the integrals 64, the products' sums ~log of their length).
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

CX = -0.75 * (3.0 / np.pi) ** (1.0 / 3.0)


def _case(n_shells, n_points, seed):
    rng = np.random.default_rng(seed)
    l = np.array([0] * n_shells if n_shells != 23 else [0, 1] * 11 + [0], dtype=np.int32)
    centre = rng.normal(size=(n_shells, 3)) * 1.5
    basis = synth.Basis(l=l, nprim=np.full(n_shells, 2, dtype=np.int32), atom=np.arange(n_shells, dtype=np.int32),
                        center=centre, exps=np.exp(rng.uniform(np.log(1e-3), np.log(1e4), 2 * n_shells)),
                        coefs=rng.uniform(0.2, 1.0, 2 * n_shells))
    pts = np.concatenate([centre, centre[:1] + 1e-9, rng.normal(size=(n_points, 3)) * 4.0])
    pts = pts[rng.permutation(len(pts))[:n_points]] if n_points <= len(pts) else pts
    grid = synth.Grid(xyz=np.ascontiguousarray(pts), w=rng.uniform(0.5, 1.5, len(pts)),
                      atom=np.zeros(len(pts), dtype=np.int32))
    nf = basis.n_functions
    C = rng.normal(size=(nf, max(1, nf // 3))) / np.sqrt(nf)
    return basis, grid, C @ C.T


@pytest.mark.parametrize("form,u", [("fp64", 512 * 2.0 ** -53), ("df32", 512 * 2.0 ** -46)])
@pytest.mark.parametrize("n_shells,n_points", [(1, 1), (16, 64), (17, 65), (23, 127), (64, 200), (65, 700), (3, 4100)])
def test_products_and_collocation_match_oracle(form, u, n_shells, n_points):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    basis, grid, P = _case(n_shells, n_points, 10 * n_shells + n_points)
    opts = dict(screen="none", eps_basis=0.0)
    if form == "df32":
        opts.update(precision="mixed", fp32_bound=0.0, ds_integrals=1, gemm="df32")
    eng = snk.Engine(basis, grid, **opts)
    eng.set_density(P)
    K = eng.build_K()
    V, _ = eng.build_Vxc(snk.XC_LDA_X)
    bound = max(eng.debug_pair_bound(a, a) for a in range(basis.n_shells))  # Cauchy-Schwarz: the largest pair
    eng.close()
    Phi = oracle.collocation(basis, grid.xyz).T
    F = P @ Phi
    a = np.abs(Phi)
    rho = (F * Phi).sum(0)
    vr = np.where(rho >= 1e-14, np.abs(4.0 / 3.0 * CX * np.maximum(rho, 0.0) ** (1.0 / 3.0)), 0.0)
    # rho itself is a sum with cancellation: its relative error enters E^rho to the power 1/3
    Fa = np.abs(P) @ a
    amp = np.where(rho >= 1e-14, np.maximum(1.0, (Fa * a).sum(0) / np.maximum(rho, 1e-14)), 0.0)
    tolV = u * float(np.max(a @ (grid.w * vr * amp * a).T))
    Vref, _ = oracle.vxc(basis, grid, P, 1)
    assert np.max(np.abs(V - Vref)) <= tolV
    tolK = u * bound * basis.n_shells * float(np.max((grid.w * Fa.max(0)) @ a.T))
    assert np.max(np.abs(K - oracle.snk_K(basis, grid, P))) <= tolK
