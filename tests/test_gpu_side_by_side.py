"""Pair lists run side by side against the same lists one after another.

A small build runs its lists on several streams with a copy of G each; the same
build cut into workspace chunks runs them one after another.  Both add the same
contributions, grouped differently: they differ by the rounding of G's sums, at
most (number of pairs) x 2^-53 of the sum of absolute values, 1e-12 of K's
largest entry here.  The form under a graph and on the caller's stream is the
same bit for bit.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

FORMS = {
    "fp64": dict(),
    "double_fp32": dict(precision="mixed", fp32_bound=0.0, ds_integrals=1, gemm="df32"),
    "mixed": dict(eps=1e-10, precision="mixed", fp32_bound=1e-3, ds_integrals=1, eps_tile=1e-11),
}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("n_atoms,n_r", [(3, 9), (7, 20)])
def test_lists_side_by_side_match_lists_in_turn(form, n_atoms, n_r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    p = synth.cluster(n_atoms, 40 + n_atoms, n_r=n_r, n_theta=4, n_phi=9, n_occ=4)

    def build(dens=1, stream=False, **kw):
        eng = snk.Engine(p.basis, p.grid, batch_max=200, **FORMS[form], **kw)
        if stream:
            eng.set_stream(torch.cuda.Stream())
        eng.set_density(p.P if dens == 1 else [p.P, 0.5 * p.P])
        K = eng.build_K()
        K = eng.build_K()
        st = eng.stats()
        eng.close()
        return np.asarray(K), st

    K, st = build()
    Kc, sc = build(workspace_bytes=1 << 20)
    assert st["n_chunks"] == 1 and sc["n_chunks"] > 1
    tol = 1e-12 * np.max(np.abs(K))
    assert np.max(np.abs(K - Kc)) <= tol
    assert np.array_equal(build(graph=1)[0], K) and np.array_equal(build(stream=True)[0], K)
    K2, _ = build(dens=2)
    # two densities share one screen (sum of |P|): more pairs kept, below the screen's threshold
    assert np.max(np.abs(K2[0] - K)) <= tol + 1e-8 and np.max(np.abs(K2[1] - 0.5 * K)) <= tol + 1e-8


def test_no_room_for_the_copies_falls_back_to_lists_in_turn():
    """An allocator that refuses the workspace with copies of G: the build runs
    its lists one after another in the smaller one, with the same K."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    p = synth.cluster(7, 47, n_r=20, n_theta=4, n_phi=9, n_occ=4)
    eng = snk.Engine(p.basis, p.grid, batch_max=200)
    eng.set_density(p.P)
    K = eng.build_K()
    with_copies = eng.stats()["workspace_bytes"]
    eng.close()
    eng = snk.Engine(p.basis, p.grid, batch_max=200)
    blocks = {}

    def alloc(nbytes):
        if nbytes >= with_copies:
            return 0
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        blocks[t.data_ptr()] = t
        return t.data_ptr()

    eng.set_allocator(alloc, lambda ptr: blocks.pop(ptr, None))
    eng.set_density(p.P)
    K1 = eng.build_K()
    assert eng.stats()["workspace_bytes"] < with_copies
    eng.close()
    assert np.max(np.abs(K1 - K)) <= 1e-12 * np.max(np.abs(K))
