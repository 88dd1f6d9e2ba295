"""Training targets of the learned correction under every preconditioner of the mixed arm: the
condensations that keep no factors of all elements give the targets of those that do."""
import numpy as np
import pytest

import oracle as O
import oracle.learned as LN
from gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _targets(n, N, precond, tc):
    from paper_1911_02366_gb300 import sc
    Q, dt, p, ctx = case(n, N, cfl=10.0, precision=sc.SC_PREC_MIXED, precond=precond, tensor_cores=tc)
    ctx.sc_set_state(Q, Q)
    ctx.sc_assemble()
    ctx.sc_condense()
    T = torch.empty(n ** 3 * len(LN.boundary_nodes(N)), 25, device="cuda")
    ctx.sc_learned_targets(T)
    return Q, dt, p, ctx, T.cpu().numpy()


@pytest.mark.parametrize("tc", [0, 1])
@pytest.mark.parametrize("precond", ["SC_PC_NONE", "SC_PC_RB_SCHUR"])
@pytest.mark.parametrize("n,N", [(1, 2), (2, 3), (4, 2), (7, 2)])  # 343 elements: more than are factorised at a time
def test_targets_do_not_depend_on_the_preconditioner(n, N, precond, tc):
    """Same S_ee, the same factorisation and products: equal to FP32 rounding of the node blocks, which
    the FP32 factors carry at 2e-3 of the largest target (as against the oracle)."""
    from paper_1911_02366_gb300 import sc
    *_, want = _targets(n, N, sc.SC_PC_BLOCK_JACOBI, tc)
    *_, ctx, T = _targets(n, N, getattr(sc, precond), tc)
    assert np.isfinite(T).all()
    assert np.max(np.abs(T - want)) <= 2e-3 * np.max(np.abs(want))


def test_targets_with_the_schur_corrected_sweep_match_the_oracle():
    """The oracle's exact targets; the solve that follows still has its preconditioner."""
    from paper_1911_02366_gb300 import sc
    n, N = 2, 3
    Q, dt, p, ctx, T = _targets(n, N, sc.SC_PC_RB_SCHUR, 0)
    S = O.condensed_operator(O.jacobian(p, Q), n, N).dense_S()
    _, To, _ = LN.features_and_targets(S, Q, n, N, 0.1, 1600.0, dt)
    assert np.max(np.abs(T - To)) <= 2e-3 * np.max(np.abs(To))
    dQ = np.zeros(Q.size)
    ctx.sc_solve(dQ)
    A, B = O.jacobian(p, Q), -O.residual(p, Q).reshape(-1)
    assert np.linalg.norm(B - A @ dQ) <= 1.01e-8 * np.linalg.norm(B)
