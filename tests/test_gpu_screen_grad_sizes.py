"""Gradient of the screen network at the edges of its sample ranges.

The samples are summed in ranges of at least 64, 16 at a time, one range per SM:
one sample, around one range, a remainder, and more ranges than SMs.  The
activations and output gradients are FP32 (relative error about 130 units of
2^-24 for the deepest sums), the sums over samples FP64, so a gradient entry is
within 2^-16 of the sum of its terms' absolute values, bounded by the largest
activation times the L1 norm of the output gradients; the loss within 2^-16.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 64, 65, 1000, 152 * 64 + 7])
def test_gradient_matches_oracle(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    rng = np.random.default_rng(n)
    w, _, _ = snk.trained_screen()
    X = rng.normal(size=(n, snk.MLP_FEATURES)).astype(np.float32) * 0.5
    Y = (-1.0 + 0.3 * rng.normal(size=n)).astype(np.float32)
    loss, g = snk.mlp_grad(w, X, Y)
    loss_ref, g_ref = oracle.mlp_loss_grad(w, X, Y)
    assert abs(loss - loss_ref) <= 2.0 ** -16 * max(loss_ref, 1e-3)
    y = oracle.mlp_forward(w, X)
    r = np.asarray(y).reshape(-1) - Y
    dy = np.sum(2.0 * np.where(r < 0, 4.0, 1.0) * np.abs(r) / n)
    # |a| and |dz / dy| are bounded by products of the layers' row sums
    scale, o = max(1.0, float(np.abs(X).max())), 0
    for n_in, n_out in ((16, 64), (64, 64), (64, 64)):
        W = np.abs(w[o:o + n_in * n_out].reshape(n_in, n_out))
        scale *= max(1.0, float(np.sqrt((W ** 2).sum(0).max())))
        o += n_in * n_out + n_out
    assert np.max(np.abs(g - g_ref)) <= 2.0 ** -16 * scale * dy * 8.0
