"""Condensed operator passes (packed rows with their couplings, split over CTAs) against S x formed
in FP64 from the assembled Jacobian blocks, at every order and for meshes that take one and several
CTAs per element."""
import numpy as np
import pytest

import oracle as O
from gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arm,n,N", [("fp64", 2, 2), ("fp64", 2, 3), ("fp64", 2, 4), ("fp64", 1, 5), ("mixed", 2, 2),
                                     ("mixed", 3, 3), ("mixed", 2, 4), ("mixed", 1, 5), ("mixed", 1, 6)])
def test_condensed_products_match_the_assembled_jacobian(arm, n, N):
    """S x = A_bb x - A_bi A_ii^-1 A_ib x through the FP64 products of sc_apply_jacobian and dense
    solves with the own blocks' interior parts.  FP64: condition of A_ii (at most 1e6) times
    rounding, 1e-9.  Mixed: FP32 blocks and interior inverses, 3e-4 of the result's scale."""
    from paper_1911_02366_gb300 import sc
    Q, dt, p, ctx = case(n, N, cfl=10.0, precision=sc.SC_PREC_MIXED if arm == "mixed" else sc.SC_PREC_FP64)
    ctx.sc_set_state(Q, Q)
    ctx.sc_assemble()
    ctx.sc_condense()
    K, ne, ni, nb = ctx.sc_sizes()
    i = np.arange(N + 1)
    inner1 = (i > 0) & (i < N)
    inner = np.repeat((inner1[:, None, None] & inner1[None, :, None] & inner1[None, None, :]).reshape(-1), 5)
    A = lambda x: ctx.sc_apply_jacobian(np.ascontiguousarray(x.reshape(-1)), np.zeros(K * ne)).reshape(K, ne)  # noqa: E731
    xb = np.random.default_rng(N).standard_normal((K, nb))
    full = np.zeros((K, ne))
    full[:, ~inner] = xb
    r = A(full)
    u = np.zeros((K, ne))
    for e in range(K):  # A_ii couples an element's interior to itself only
        Aii = np.zeros((ni, ni))
        if n > 1:
            Aii = ctx.sc_get_jacobian_block(e, e)[np.ix_(inner, inner)]
        else:
            for c in range(ni):
                x = np.zeros((K, ne))
                x[0, np.flatnonzero(inner)[c]] = 1.0
                Aii[:, c] = A(x)[0, inner]
        u[e, inner] = np.linalg.solve(Aii, r[e, inner])
    want = (r - A(u))[:, ~inner].reshape(-1)
    y = torch.zeros(K * nb, dtype=torch.float64, device="cuda")
    ctx.sc_condensed_matvec(torch.tensor(xb.reshape(-1), device="cuda"), y)
    tol = 1e-9 if arm == "fp64" else 3e-4
    assert np.abs(y.cpu().numpy() - want).max() <= tol * np.abs(want).max()
