"""FP64 Boys seeds half way between the table's nodes (spacing 1/12), on both
sides of T = 50, and for T so small that 2T by the exponent is not exact.

Tolerance: the polynomial's and e^x's truncations are below 3e-16, the chain
has at most 16 roundings of 1.1e-16, together 2.1e-15; the oracle's F_n are
pinned to 1e-14 relative."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOL = 1.3e-14


@pytest.mark.parametrize("nmax", range(5))
def test_boys_between_nodes(nmax):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    mid = (np.arange(600) + 0.5) / 12.0
    T = np.concatenate([mid, np.nextafter(mid, 0.0), np.arange(600) / 12.0,
                        [np.nextafter(50.0, 0.0), 50.0, np.nextafter(50.0, 60.0)]])
    ref = np.array([oracle.boys(nmax, t) for t in T])
    d = snk.debug_boys(T, nmax)
    assert np.max(np.abs(d - ref) / ref) <= TOL
    tiny = np.array([0.0, 5e-324, 1e-310, 2.3e-308, 1e-200, 1e-30])
    ref0 = 1.0 / (2.0 * np.arange(nmax + 1) + 1.0)
    assert np.max(np.abs(snk.debug_boys(tiny, nmax) / ref0 - 1.0)) <= TOL
