"""No sample is lost at the edges of the gradient's sample ranges.

With every label equal to its prediction and one label off by 10,000, the gradient
less the gradient without that error is the one sample's share.  The sample sits
at every place where the sum over samples is cut: the first and last of a range, of a
step of 16 samples, of a block of 128, the last of all, for up to the full 152 ranges
(n = 9,728 and 12,160, and 7 fewer).

Tolerance per entry, from an FP64 backward pass of the one sample: a gradient entry
is a product of an activation and an output gradient, chains of at most 130 FP32
roundings between them, 130 x 2^-24 of the product of the two chains run on absolute
values; the prediction's own rounding, 130 x 2^-24 of its chain on absolute values,
relative to 10,000 (four times that, when it counts as an under-prediction); and the
rounding of the two gradients.  A lost sample changes every entry by its whole value;
the test asserts that their norm is ten times the tolerance's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 130 * 2.0 ** -24
ERROR = 1e4
LAYERS = ((16, 64), (64, 64), (64, 64), (64, 1))


def _layers(w):
    out, o = [], 0
    for n_in, n_out in LAYERS:
        W = w[o:o + n_in * n_out].astype(np.float64).reshape(n_in, n_out)
        o += n_in * n_out
        out.append((W, w[o:o + n_out].astype(np.float64)))
        o += n_out
    return out


def _forward(layers, X):
    """Activations of every layer, and the same chains on absolute values."""
    a, b = [X], [np.abs(X)]
    for k, (W, bias) in enumerate(layers):
        z = a[-1] @ W + bias
        a.append(np.maximum(z, 0.0) if k < 3 else z)
        b.append(b[-1] @ np.abs(W) + np.abs(bias))
    return a, b


def _gradient(layers, x, dy):
    """Gradient of one sample and its bound on absolute values, weights then biases layer by layer."""
    a, b = _forward(layers, x[None])
    d, e = np.array([[dy]]), np.abs(np.array([[dy]]))
    g, m = [None] * 4, [None] * 4
    for k in (3, 2, 1, 0):
        W = layers[k][0]
        g[k] = np.concatenate([(a[k].T @ d).ravel(), d.ravel()])
        m[k] = np.concatenate([(b[k].T @ e).ravel(), e.ravel()])
        if k:
            d, e = (d @ W.T) * (a[k] > 0), (e @ np.abs(W).T) * (a[k] > 0)
    return np.concatenate(g), np.concatenate(m)


@pytest.mark.parametrize("n", [1, 16, 17, 64, 65, 129, 1000, 152 * 64, 152 * 80, 152 * 80 - 7])
def test_every_edge_sample_counts(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_14280_gb300 as snk
    rng = np.random.default_rng(n)
    w, _, _ = snk.trained_screen()
    X = (0.5 * rng.normal(size=(n, snk.MLP_FEATURES))).astype(np.float32)
    layers = _layers(w)
    a, b = _forward(layers, X.astype(np.float64))
    pred = np.asarray(snk.mlp_eval(w, X)).reshape(-1)
    loss0, g0 = (np.float64(v) for v in snk.mlp_grad(w, X, pred))
    ranges = min(152, -(-n // 64))
    klen = -(-(-(-n // ranges)) // 16) * 16
    last = (n - 1) // klen * klen  # the last range's first sample
    for s in sorted({k for k in (0, 15, 16, klen - 1, klen, 127, 128, last - 1, last, (n - 1) // 16 * 16, n - 2, n - 1)
                     if 0 <= k < n}):
        Y = pred.copy()
        Y[s] -= np.float32(ERROR)  # over-predicted: c = 1, dL/dy = 2 r / n
        loss, g = snk.mlp_grad(w, X, Y)
        r = float(pred[s] - Y[s])
        ref, mag = _gradient(layers, X[s].astype(np.float64), 2.0 * r / n)
        off = 8.0 * U * b[4][s, 0] / ERROR  # the prediction's rounding, with and without the error
        tol = (U + off) * mag + 2.0 ** -23 * (np.abs(g) + np.abs(g0))
        assert np.linalg.norm(tol) <= 0.1 * np.linalg.norm(ref), "the tolerance would hide a lost sample"
        assert np.all(np.abs((g - g0) - ref) <= tol), f"sample {s} of {n}"
        assert abs((loss - loss0) * n / r ** 2 - 1.0) <= 2.0 * off + 2.0 ** -20
