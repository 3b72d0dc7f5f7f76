"""Algorithmic flops that the statistics report, on a molecule of one uncontracted
shell (one shell pair, one primitive pair): the FP32 tier counts the recursion that
its pp and dd classes run, the FP64 form the contraction.  Counts by hand from the
generated code's operations: T and Boys function 8 + (3 + 2 L), then recursion + HRR or
contraction + contracted recursion, then 2 n_a n_b."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l,fp32,fp64", [(0, 8 + 1 + 1 + 2, 8 + 1 + 1 + 2), (1, 8 + 7 + 54 + 18 + 18, 8 + 7 + 13 + 66 + 18),
                                         (2, 8 + 11 + 268 + 158 + 72, 8 + 11 + 45 + 503 + 72)])
def test_flops_of_one_pair(l, fp32, fp64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    rng = np.random.default_rng(l)
    basis = synth.Basis(l=np.array([l], dtype=np.int32), nprim=np.array([1], dtype=np.int32),
                        atom=np.array([0], dtype=np.int32), center=np.zeros((1, 3)), exps=np.array([0.7]),
                        coefs=np.array([1.0]))
    q = 37
    grid = synth.Grid(xyz=rng.normal(size=(q, 3)), w=np.ones(q), atom=np.zeros(q, dtype=np.int32))
    for opts, key, want in ((dict(eps_E=0.0, eps_K=0.0, precision="mixed", fp32_bound=1e30), "flops_fp32", fp32),
                            (dict(screen="none"), "integral_flops", fp64)):
        eng = snk.Engine(basis, grid, eps_basis=0.0, **opts)
        eng.set_density(np.eye(basis.n_functions))
        listed = eng.stats()[key]
        eng.build_K()
        assert listed == want * q and eng.stats()[key] == want * q
        eng.close()
