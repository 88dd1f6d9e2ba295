"""Gram-Schmidt sweeps over more vectors than 48 KB of shared memory hold the sums of (171 and more)."""
import numpy as np
import pytest

import oracle as O
from gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N", [(2, 3), (3, 2)])  # 2240 and 3645 (odd: no 16-byte pieces) boundary values
def test_one_cycle_of_more_than_171_vectors(n, N):
    """Without a preconditioner GMRES needs several hundred iterations, the first 400 in one cycle.  The
    residual is recomputed with the oracle; rounding of the FP64 operator allows 1e-12 of |B| on top."""
    from paper_1911_02366_gb300 import sc
    Q, dt, p, ctx = case(n, N, cfl=2.0, precond=sc.SC_PC_NONE, gmres_restart=400, rel_tol=1e-8, gmres_max_iters=4000)
    ctx.sc_set_state(Q, Q)
    ctx.sc_assemble()
    ctx.sc_condense()
    dQ = np.zeros(Q.size)
    st = ctx.sc_solve(dQ)
    assert st["gmres_iters"] > 171, st
    B = -O.residual(p, Q).reshape(-1)
    r = B - O.jvp(p, Q, dQ.reshape(Q.shape)).reshape(-1)
    assert np.linalg.norm(r) <= (1e-8 + 1e-12) * np.linalg.norm(B), st
