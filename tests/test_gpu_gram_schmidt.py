"""Gram-Schmidt sweeps through the solvers that use them: odd vector lengths (no 16-byte pieces), a
basis longer than a default block's shared memory, and one vector per cycle."""
import numpy as np
import pytest

import oracle as O
from gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,cfg", [(3, 2, dict(outer_krylov=8, inner_iters=10, arm="mixed")),  # 27 x 135 dofs: odd
                                     (2, 3, dict(gmres_restart=1, rel_tol=1e-6)), (2, 3, dict(gmres_restart=400)),
                                     (4, 2, dict(gmres_restart=7))])
def test_solves_reach_the_tolerance_they_are_given(n, N, cfg):
    """The residual is recomputed with the oracle; rounding of the FP64 operator allows 1e-12 of |B| on top."""
    from paper_1911_02366_gb300 import sc
    cfg = dict(cfg)
    tol = cfg.pop("rel_tol", 1e-11)
    arm = sc.SC_PREC_MIXED if cfg.pop("arm", "fp64") == "mixed" else sc.SC_PREC_FP64
    Q, dt, p, ctx = case(n, N, cfl=2.0, precision=arm, rel_tol=tol, gmres_max_iters=4000, max_refine=20, **cfg)
    ctx.sc_set_state(Q, Q)
    ctx.sc_assemble()
    ctx.sc_condense()
    dQ = np.zeros(Q.size)
    st = ctx.sc_solve(dQ)
    B = -O.residual(p, Q).reshape(-1)
    r = B - O.jvp(p, Q, dQ.reshape(Q.shape)).reshape(-1)
    assert np.linalg.norm(r) <= (tol + 1e-12) * np.linalg.norm(B), st
