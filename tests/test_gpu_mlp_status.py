"""A tensor-core wait of the network's forward pass that runs out: the entry points report it, and training
leaves the parameters alone.  The library is built once more with waits that give up at once; its
kernel still lets its products finish before it returns, so the device stays usable."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    from paper_1911_02366_gb300 import build as b
    out = str(tmp_path_factory.mktemp("mlp") / "libmlp.so")
    subprocess.run([b.nvcc(), *b.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-shared",
                    "-DSC_MLP_WAIT_POLLS=-1", os.path.join(b.CSRC, "sc_mlp.cu"), "-o", out], check=True)
    return ctypes.CDLL(out)


def test_expired_waits_are_errors(impatient):
    from paper_1911_02366_gb300 import sc
    rng = np.random.default_rng(0)
    net = sc.MLP(rng.standard_normal(sc.MLP_NW).astype(np.float32) * 0.1, np.zeros(sc.MLP_NB, np.float32))
    n = 300
    X = torch.randn(n, 128, device="cuda")
    T = torch.randn(n, 25, device="cuda")
    Y = torch.zeros(n, 25, device="cuda")
    vp = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    torch.cuda.synchronize()
    assert impatient.sc_mlp_forward(vp(net.Wh), vp(net.b), vp(X), n, vp(Y), None, None) == sc.SC_ERR_CUDA
    assert bool(torch.isnan(Y).all())
    W, m, v = net.W.clone(), torch.zeros(sc.MLP_NW + sc.MLP_NB, device="cuda"), torch.zeros(sc.MLP_NW + sc.MLP_NB, device="cuda")
    b, Wh = net.b.clone(), net.Wh.clone()
    step, loss = ctypes.c_int(0), (ctypes.c_float * 2)()
    torch.cuda.synchronize()
    s = impatient.sc_mlp_train(vp(net.W), vp(net.Wh), vp(net.b), vp(m), vp(v), ctypes.byref(step), vp(X), vp(T), n, 2, 128,
                               ctypes.c_float(1e-3), ctypes.c_uint64(1), loss, None)
    assert s == sc.SC_ERR_CUDA and step.value == 0
    assert torch.equal(W, net.W) and torch.equal(b, net.b) and torch.equal(Wh, net.Wh) and not bool(m.any())
    net.forward(X, Y)  # the library's own waits are met
    assert bool(torch.isfinite(Y).all())
