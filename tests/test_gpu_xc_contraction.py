"""V^xc with shells of more than four primitives, whose exponentials the collocation
forms one by one instead of group by group.

The same functions written with 3 primitives and with each of them twice at half
the coefficient (6 primitives) have the same X and gradients up to rounding, so V
and E_xc agree to 512 u of the sums of the products' absolute values, here 1e-12 of
V's largest entry; both match the oracle to the plain path's 1e-10 (the FP64 and
double-FP32 tiles).  s, p and d shells alone and together, some sharing exponents."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _basis(ls, copies, xyz):
    l, atom, center, exps, coefs = [], [], [], [], []
    for a, x in enumerate(xyz):
        for k, la in enumerate(ls):
            l.append(la)
            atom.append(a)
            center.append(x)
            e = 0.15 * (1.0 + 0.3 * (k // 2)) * 4.0 ** np.arange(3)
            exps += list(np.repeat(e, copies))
            coefs += list(np.repeat([0.5, 0.4, 0.3], copies) / copies)
    return synth.Basis(l=np.array(l, dtype=np.int32), nprim=np.full(len(l), 3 * copies, dtype=np.int32),
                       atom=np.array(atom, dtype=np.int32), center=np.array(center), exps=np.array(exps),
                       coefs=np.array(coefs))


@pytest.mark.parametrize("form", ["fp64", "df32"])
@pytest.mark.parametrize("ls", [(0,), (1,), (2,), (0, 1, 2, 2)])
def test_many_primitives_match_few(ls, form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    rng = np.random.default_rng(31)
    xyz = np.array([[0.0, 0.1, -0.2], [1.9, -0.4, 0.3], [-0.7, 1.6, 1.1]])
    grid = synth.Grid(xyz=np.concatenate([xyz, rng.normal(size=(700, 3)) * 2.0]), w=rng.uniform(0.01, 0.05, 703),
                      atom=np.zeros(703, dtype=np.int32))
    opts = dict(eps_basis=0.0)
    if form == "df32":
        opts.update(precision="mixed", gemm="df32")
    got = {}
    for copies in (1, 2):
        basis = _basis(ls, copies, xyz)
        C = np.random.default_rng(5).normal(size=(basis.n_functions, 3)) / np.sqrt(basis.n_functions)
        P = C @ C.T
        eng = snk.Engine(basis, grid, **opts)
        eng.set_density(P)
        for fun in (oracle.XC_LDA_X, oracle.XC_PBE):
            V, E = eng.build_Vxc(fun)
            Vr, Er = oracle.vxc(basis, grid, P, fun)
            assert np.max(np.abs(V - Vr)) <= 1e-10 and abs(E - Er) <= 1e-10
            got[copies, fun] = V, E
        eng.close()
    for fun in (oracle.XC_LDA_X, oracle.XC_PBE):
        (V1, E1), (V2, E2) = got[1, fun], got[2, fun]
        assert np.max(np.abs(V1 - V2)) <= 1e-12 * np.max(np.abs(V1)) and abs(E1 - E2) <= 1e-12 * abs(E1)
