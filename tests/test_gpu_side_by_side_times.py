"""Phase times of builds that run their pair lists side by side: every list's time
goes to its own tier and class.

The tiers' times add up to the phase (inside ms_build), a class without pairs has
none, and the FP32 tier's work over its time stays below the FP32 pipes' rate
(152 SMs x 128 lanes x 2 flops x 2.07 GHz = 80.5 TFLOP/s), which a time that holds
only the gap between two events exceeds many times over."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MIXED = dict(eps=1e-10, precision="mixed", fp32_bound=1e-3, ds_integrals=1, eps_tile=1e-11)


@pytest.mark.parametrize("share", [None, 0.3, 0.04])
@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_every_list_has_its_own_time(form, share):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    p = synth.cluster(12, 61, n_r=40, n_theta=5, n_phi=12, n_occ=8)
    opts = dict(MIXED) if form == "mixed" else {}

    def build(**kw):
        eng = snk.Engine(p.basis, p.grid, **opts, **kw)
        eng.set_density(p.P)
        for _ in range(3):
            eng.build_K()
        st = eng.stats()
        eng.close()
        return st

    st = build()
    if share is not None:
        st = build(workspace_bytes=int(share * st["workspace_bytes"]))
    hi, lo = np.array(st["ms_integrals_class"]), np.array(st["ms_integrals_class_fp32"])
    assert abs(hi.sum() - st["ms_integrals"]) <= 1e-9 + 1e-6 * st["ms_integrals"]
    assert abs(lo.sum() - st["ms_integrals_fp32"]) <= 1e-9 + 1e-6 * st["ms_integrals_fp32"]
    assert st["ms_integrals"] + st["ms_integrals_fp32"] <= st["ms_build"]
    assert np.all((hi > 0.0) == (np.array(st["integrals_class"]) > 0.0))
    if form == "mixed":
        assert st["pairs_kept_fp32"] > 0 and np.count_nonzero(lo) > 1
        assert st["flops_fp32"] / (st["ms_integrals_fp32"] * 1e-3) < 80.5e12
    else:
        assert np.all(lo == 0.0) and st["ms_integrals_fp32"] == 0.0
