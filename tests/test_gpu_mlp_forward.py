"""The tensor-core forward pass at the edges of its 128-sample tiles, with unaligned parameters and
inputs, and with infinities and NaN, against the network in 64 bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _network(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    W = torch.cat([(r(256, 128) * 0.125).reshape(-1), (r(256, 256) * 0.088).reshape(-1), (r(25, 256) * 0.06).reshape(-1)])
    return W.cpu().numpy(), (0.1 * r(537)).cpu().numpy(), g


def _exact(net, X):
    W = net.Wh.view(torch.bfloat16).double()
    b = net.b.double()
    z1 = X.double() @ W[:32768].view(256, 128).T + b[:256]
    z2 = torch.relu(z1) @ W[32768:98304].view(256, 256).T + b[256:512]
    return z1, z2, torch.relu(z2) @ W[98304:].view(25, 256).T + b[512:]


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("shift", [0, 1])
def test_forward_matches_the_network_in_64_bits(n, shift):
    """Sums of at most 256 exact products in FP32: n_k eps of the absolute sums at worst; the sums'
    typical size is a tenth of that, so 256 * 2^-24 = 1.5e-5 of the largest output bounds both layers."""
    from paper_1911_02366_gb300 import sc
    W, b, g = _network(3 + n)
    net = sc.MLP(W, b)
    store = torch.empty(n * 128 + 4, device="cuda")
    X = store[shift:shift + n * 128].view(n, 128)
    X.copy_(torch.randn(n, 128, device="cuda", generator=g) * torch.logspace(-6, 3, 128, device="cuda")[None, :] * 1e-2)
    if shift:  # parameters off the 16-byte grid too
        Wh = torch.empty(net.Wh.numel() + 1, dtype=torch.int16, device="cuda")
        Wh[1:] = net.Wh
        net.Wh = Wh[1:]
    Y = torch.empty(n, 25, device="cuda")
    cache = torch.empty(4 * n * 256 + 1, device="cuda")[shift:shift + 4 * n * 256]
    net.forward(X, Y, cache)
    z1, z2, y = _exact(net, X)
    parts = cache.view(4, n, 256).double()
    for got, want in ((parts[0], z1), (parts[1], torch.relu(z1)), (parts[2], z2), (parts[3], torch.relu(z2)), (Y.double(), y)):
        assert float((got - want).abs().max()) <= 1.5e-5 * float(want.abs().max())
    Y2 = torch.empty_like(Y)
    net.forward(X, Y2)
    assert torch.equal(Y, Y2)


def test_non_finite_inputs_stay_in_their_samples():
    from paper_1911_02366_gb300 import sc
    W, b, g = _network(9)
    net = sc.MLP(W, b)
    X = torch.randn(200, 128, device="cuda", generator=g)
    Y0 = net.forward(X, torch.empty(200, 25, device="cuda")).clone()
    bad = X.clone()
    bad[3, 7], bad[130, 100], bad[199, 0] = float("nan"), float("inf"), 3.4e38
    cache = torch.empty(4, 200, 256, device="cuda")
    Y = net.forward(bad, torch.empty(200, 25, device="cuda"), cache)
    keep = torch.ones(200, dtype=torch.bool, device="cuda")
    keep[[3, 130, 199]] = False
    assert torch.equal(Y[keep], Y0[keep])
    z1 = cache[0]
    assert bool(torch.isnan(z1[3]).all())
    w = net.Wh.view(torch.bfloat16).float()[:32768].view(256, 128)
    assert torch.equal(z1[130], torch.where(w[:, 100] > 0, float("inf"), -float("inf")))
    big = bad[199].double() @ w.double().T + net.b[:256].double()  # the largest finite values: no early overflow
    fits = big.abs() < 3e38
    assert float((z1[199].double() - big).abs()[fits].max()) <= 1.5e-5 * float(big.abs().max())
