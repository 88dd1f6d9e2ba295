"""The network's forward pass with infinite and NaN weights: as sums of products, term by term."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(net, X):
    """Pre- and post-activations and outputs in 64 bits; ReLU as max(z, 0) with NaN -> 0, as in FP32 fmaxf."""
    W = net.Wh.view(torch.bfloat16).double().cpu().numpy()
    b = net.b.double().cpu().numpy()
    W1, W2, W3 = W[:32768].reshape(256, 128), W[32768:98304].reshape(256, 256), W[98304:].reshape(25, 256)
    with np.errstate(invalid="ignore"):
        z1 = X.double().cpu().numpy() @ W1.T + b[:256]
        h1 = np.fmax(z1, 0.0)
        z2 = h1 @ W2.T + b[256:512]
        h2 = np.fmax(z2, 0.0)
        return [z1, h1, z2, h2, h2 @ W3.T + b[512:]]


@pytest.mark.parametrize("where", [((0, 5, 7, np.inf),), ((0, 200, 127, -np.inf), (2, 3, 9, np.inf)), ((1, 17, 33, np.inf),),
                                   ((1, 255, 255, -np.inf),), ((2, 24, 255, np.inf),), ((2, 0, 0, -np.inf),),
                                   ((1, 4, 4, np.nan),)])
def test_infinite_weights_give_the_infinities_of_the_products(where):
    """Inputs that BF16 holds exactly, 0 among them, and inputs it does not; finite values to FP32
    accumulation (256 terms, 1.5e-5 of the largest), the others exactly."""
    from paper_1911_02366_gb300 import sc
    rng = np.random.default_rng(11)
    W = np.concatenate([(rng.standard_normal(s) * f).reshape(-1)
                        for s, f in (((256, 128), 0.125), ((256, 256), 0.088), ((25, 256), 0.06))]).astype(np.float32)
    for layer, row, col, value in where:
        W[(0, 32768, 98304)[layer] + row * (128, 256, 256)[layer] + col] = value
    net = sc.MLP(W, 0.1 * rng.standard_normal(537).astype(np.float32))
    n = 200
    X = torch.tensor(rng.standard_normal((n, 128)), dtype=torch.float32, device="cuda")
    X[::3] = torch.round(X[::3] * 4) / 4
    X[5] = 1.0
    X[6] = 0.0
    Y = torch.empty(n, 25, device="cuda")
    cache = torch.empty(4, n, 256, device="cuda")
    net.forward(X, Y, cache)
    want = _reference(net, X)
    for name, g, w in zip(("z1", "h1", "z2", "h2", "y"), [*cache, Y], want):
        g = g.double().cpu().numpy()
        fin = np.isfinite(w)
        assert np.array_equal(np.isnan(g), np.isnan(w)), name
        assert np.array_equal(g[~fin & ~np.isnan(w)], w[~fin & ~np.isnan(w)]), name
        if fin.any():
            assert np.abs(g[fin] - w[fin]).max() <= 1.5e-5 * np.abs(w[fin]).max(), name
