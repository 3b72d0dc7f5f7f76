"""FP64 pairs of uncontracted shells take the recursion for their one primitive pair,
all others are contracted first: the two on the same functions.

Every primitive written twice with half the coefficient is the same basis with four
primitive pairs per pair of shells, and a basis with every second shell written so
has lists that mix both forms.  Both K are sums of the same terms in chains of at
most 64 roundings per block, so they agree to 64 u times the sum of absolute values,
below 1e-12 of K's largest entry here (the bound of the side-by-side comparison)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _basis(rng, n_atoms, twice):
    l, atom, center, exps, coefs, nprim = [], [], [], [], [], []
    xyz = rng.uniform(-2.5, 2.5, size=(n_atoms, 3))
    for a in range(n_atoms):
        for la, e in ((0, 0.4), (1, 0.9), (1, 0.3), (2, 0.7), (2, 0.25)):
            k = 2 if twice == "all" or (twice == "some" and len(l) % 2) else 1
            l.append(la)
            atom.append(a)
            center.append(xyz[a])
            nprim.append(k)
            exps += [e * (1.0 + 0.1 * a)] * k
            coefs += [1.0 / k] * k
    return synth.Basis(l=np.array(l, dtype=np.int32), nprim=np.array(nprim, dtype=np.int32),
                       atom=np.array(atom, dtype=np.int32), center=np.array(center), exps=np.array(exps),
                       coefs=np.array(coefs))


@pytest.mark.parametrize("n_atoms,n_points", [(1, 1), (2, 129), (4, 1500)])
@pytest.mark.parametrize("n_dens", [1, 2])
def test_recursion_and_contraction_agree(n_atoms, n_points, n_dens):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    K = {}
    for twice in ("none", "some", "all"):
        rng = np.random.default_rng(17 + n_atoms)
        basis = _basis(rng, n_atoms, twice)
        grid = synth.Grid(xyz=rng.normal(size=(n_points, 3)) * 2.5, w=rng.uniform(0.2, 1.0, n_points),
                          atom=np.zeros(n_points, dtype=np.int32))
        P = rng.normal(size=(basis.n_functions,) * 2)
        P = P + P.T
        eng = snk.Engine(basis, grid, eps_basis=0.0, screen="none")
        eng.set_density(P if n_dens == 1 else [P, P @ P])
        K[twice] = np.asarray(eng.build_K())
        eng.close()
    for twice in ("some", "all"):
        for a, b in zip(np.atleast_3d(K[twice].T).T, np.atleast_3d(K["none"].T).T):
            assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
