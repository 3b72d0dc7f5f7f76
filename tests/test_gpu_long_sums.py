"""Double-FP32 sums over long runs of pairs, against the FP64 form.

2,000 single-primitive s shells, a positive density and one point: G_a of the last
shells is one run of about 2,000 terms of one sign, and K's entries between two
such shells are two G values times the collocation, with nothing to average over.

Tolerance: a renormalised sum rounds lo and the result to 2^-49 of the running sum,
each term adds its product's and its block's rounding of the same size: four
independent roundings of up to 2^-49 a term, sqrt(4 n / 3) 2^-49 = 9e-14 rms for a sum
of n = 2,000 terms, and an entry of K is the mean of two such sums.  Twice the mean's
value is allowed, 1.3e-13; sums that are never renormalised are off by 3.5e-13 rms
each, 2.5e-13 the mean of two."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_rms_error_of_long_runs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    n = 2000
    rng = np.random.default_rng(3)
    center = rng.uniform(-1.0, 1.0, size=(n, 3))
    basis = synth.Basis(l=np.zeros(n, dtype=np.int32), nprim=np.ones(n, dtype=np.int32),
                        atom=np.arange(n, dtype=np.int32), center=center, exps=rng.uniform(0.1, 0.4, n),
                        coefs=np.ones(n))
    v = rng.uniform(0.5, 1.0, n)
    P = np.outer(v, v)
    grid = synth.Grid(xyz=np.array([[0.1, 0.2, -0.3]]), w=np.array([1.0]), atom=np.zeros(1, dtype=np.int32))
    K = {}
    for name, opts in (("fp64", dict()), ("ds", dict(precision="mixed", fp32_bound=0.0, ds_integrals=1))):
        eng = snk.Engine(basis, grid, eps_basis=0.0, screen="none", **opts)
        eng.set_density(P)
        K[name] = np.asarray(eng.build_K())
        eng.close()
    last = slice(n - 100, n)
    rel = (K["ds"][last, last] / K["fp64"][last, last] - 1.0)
    assert np.min(K["fp64"][last, last]) > 0.0
    assert np.sqrt(np.mean(rel ** 2)) <= 2.0 * np.sqrt(4.0 * n / 3.0 / 2.0) * 2.0 ** -49
