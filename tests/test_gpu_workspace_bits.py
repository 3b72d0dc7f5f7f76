"""K is the same bit for bit whatever the workspace holds: all copies of G at once, some
of them at a time, one beside the sum, one chunk or many, and when the allocator
refuses the larger plans (once: later densities do not ask again)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

FORMS = {
    "fp64": dict(),
    "double_fp32": dict(precision="mixed", fp32_bound=0.0, ds_integrals=1, gemm="df32"),
    "mixed_fp64_products": dict(eps=1e-10, precision="mixed", fp32_bound=1e-3, ds_integrals=1, eps_tile=1e-11),
    "mixed_split": dict(eps=1e-10, precision="mixed", fp32_bound=1e-3, ds_integrals=1, gemm="split", eps_tile=1e-11),
}


def _snk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    return torch, snk


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("n_dens", [1, 2])
def test_any_workspace_gives_the_same_bits(form, n_dens):
    _, snk = _snk()
    p = synth.cluster(6, 46, n_r=20, n_theta=4, n_phi=9, n_occ=4)

    def build(**kw):
        eng = snk.Engine(p.basis, p.grid, batch_max=200, **FORMS[form], **kw)
        eng.set_density(p.P if n_dens == 1 else [p.P, 0.5 * p.P @ p.P])
        K = np.asarray(eng.build_K()).copy()
        st = eng.stats()
        eng.close()
        return K, st

    K, st = build()
    full, chunks = st["workspace_bytes"], set()
    for share in (1.2, 0.8, 0.6, 0.45, 0.3, 0.2, 0.12, 0.06, 0.02):
        Kw, sw = build(workspace_bytes=int(share * full))
        chunks.add(sw["n_chunks"])
        assert np.array_equal(Kw, K), f"{share} of the workspace, {sw['n_chunks']} chunks"
    assert min(chunks) == 1 and max(chunks) > 2


def test_batch_handle_and_graph():
    _, snk = _snk()
    ps = [synth.cluster(n, 50 + n, n_r=16, n_theta=4, n_phi=9, n_occ=3) for n in (3, 5, 4)]

    def build(**kw):
        eng = snk.Engine([p.basis for p in ps], [p.grid for p in ps], batch_max=200, **FORMS["double_fp32"], **kw)
        eng.set_density([p.P for p in ps])
        K = [np.asarray(k).copy() for k in eng.build_K()]
        w = eng.stats()["workspace_bytes"]
        eng.close()
        return K, w

    K, full = build()
    for kw in (dict(graph=1), dict(workspace_bytes=full // 2), dict(workspace_bytes=full // 4, graph=1),
               dict(workspace_bytes=full // 20)):
        assert all(np.array_equal(a, b) for a, b in zip(build(**kw)[0], K)), kw


def test_refused_plans_keep_the_bits_and_are_not_tried_again():
    torch, snk = _snk()
    p = synth.cluster(6, 46, n_r=20, n_theta=4, n_phi=9, n_occ=4)
    eng = snk.Engine(p.basis, p.grid, batch_max=200)
    eng.set_density(p.P)
    K = np.asarray(eng.build_K()).copy()
    full = eng.stats()["workspace_bytes"]
    eng.close()
    for most in (0.9 * full, 0.5 * full, 0.25 * full, 0.17 * full):
        blocks, refused = {}, []

        def alloc(nbytes):
            if nbytes > most:
                refused.append(nbytes)
                return 0
            t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
            blocks[t.data_ptr()] = t
            return t.data_ptr()

        eng = snk.Engine(p.basis, p.grid, batch_max=200)
        eng.set_allocator(alloc, lambda ptr: blocks.pop(ptr, None))
        eng.set_density(p.P)
        assert refused and np.array_equal(np.asarray(eng.build_K()), K)
        n = len(refused)
        eng.set_density(p.P)
        assert len(refused) == n and np.array_equal(np.asarray(eng.build_K()), K)
        eng.close()


def test_no_copies_for_lists_without_pairs():
    """With every pair in the FP32 tier the copies of G for ranges of the FP64 lists
    would stay zero: the workspace holds one per lane (3), not up to 24 (about a fifth
    of the FP64 form's doubles; half is allowed for X and the FP32 copy of F)."""
    _, snk = _snk()
    p = synth.cluster(4, 44, n_r=20, n_theta=4, n_phi=9, n_occ=4)
    held = {}
    for name, opts in (("fp64", dict()), ("fp32", dict(eps_E=0.0, eps_K=0.0, precision="mixed", fp32_bound=1e30))):
        eng = snk.Engine(p.basis, p.grid, batch_max=200, **opts)
        eng.set_density(p.P)
        eng.build_K()
        held[name] = eng.stats()["workspace_bytes"]
        eng.close()
    assert held["fp32"] < 0.5 * held["fp64"]


@pytest.mark.parametrize("kw", [dict(), dict(graph=1), dict(share=0.3), dict(share=0.05, graph=1)])
def test_learned_screen_side_by_side(kw):
    """The learned screen rewrites the lists before they are cut: the same bits with all
    copies, in a graph, and group by group; two densities loaded one after another."""
    _, snk = _snk()
    p = synth.cluster(9, 49, n_r=20, n_theta=4, n_phi=9, n_occ=5)
    w, skip, meta = snk.trained_screen()
    opts = dict(FORMS["mixed_split"], screen="learned", learned_skip=skip, learned_fp32=meta["fp32_threshold"])

    def build(**kw):
        eng = snk.Engine(p.basis, p.grid, batch_max=200, **opts, **kw)
        eng.screen_load(w)
        K = []
        for P in (p.P, 0.01 * p.P, p.P):
            eng.set_density(P)
            K.append(np.asarray(eng.build_K()).copy())
        st = eng.stats()
        eng.close()
        return K, st

    K, st = build()
    assert st["pairs_learned_skipped"] > 0 and np.array_equal(K[0], K[2])
    kw = dict(kw)
    if "share" in kw:
        kw["workspace_bytes"] = int(kw.pop("share") * st["workspace_bytes"])
    assert all(np.array_equal(a, b) for a, b in zip(build(**kw)[0], K))
