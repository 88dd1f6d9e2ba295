"""Block solves in the form of one CTA per element (partitioned inverses), which larger FP64 blocks and the
largest FP32 ones take between the meshes of inverted triangles and those of a warp per element, and
the FP64 LU of many blocks: against S_ee in FP64 from the assembled own blocks."""
import numpy as np
import pytest

import oracle as O
from gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _system(arm, n, N, precond):
    from paper_1911_02366_gb300 import sc
    Q, dt, p, ctx = case(n, N, cfl=10.0, precision=sc.SC_PREC_MIXED if arm == "mixed" else sc.SC_PREC_FP64, precond=precond)
    ctx.sc_set_state(Q, Q)
    ctx.sc_assemble()
    ctx.sc_condense()
    return ctx


def _schur_block(ctx, e, N):
    A = ctx.sc_get_jacobian_block(e, e)
    i = np.arange(N + 1)
    i1 = (i > 0) & (i < N)
    m = np.repeat((i1[:, None, None] & i1[None, :, None] & i1[None, None, :]).reshape(-1), 5)
    return A[np.ix_(~m, ~m)] - A[np.ix_(~m, m)] @ np.linalg.solve(A[np.ix_(m, m)], A[np.ix_(m, ~m)])


def _apply(f, v):
    y = torch.zeros(v.size, dtype=torch.float64, device="cuda")
    f(torch.tensor(v, device="cuda"), y)
    return y.cpu().numpy()


# the last mesh of inverted triangles and the first of the CTA form, either side of the FP64 lines; 512 blocks
# of n_b = 130, 280 and 490 also take the LU of one CTA per block
@pytest.mark.parametrize("arm,n,N", [("fp64", 8, 2), ("fp64", 10, 3), ("fp64", 11, 3), ("fp64", 7, 4), ("fp64", 8, 4),
                                     ("fp64", 6, 5), ("fp64", 7, 5), ("mixed", 11, 5), ("mixed", 12, 5)])
def test_block_jacobi_in_every_form(arm, n, N):
    """Backward error of S_ee z_e = v_e; bounds as for the small meshes (FP64 1e-12, TF32 products 2e-3)."""
    from paper_1911_02366_gb300 import sc
    ctx = _system(arm, n, N, sc.SC_PC_BLOCK_JACOBI)
    K, _, _, nb = ctx.sc_sizes()
    v = np.random.default_rng(N).standard_normal(K * nb)
    z = _apply(ctx.sc_precond_apply, v)
    for e in (0, K // 2, K - 1):
        S, ze, ve = _schur_block(ctx, e, N), z[e * nb:(e + 1) * nb], v[e * nb:(e + 1) * nb]
        scale = np.abs(S).sum(axis=1).max() * np.abs(ze).max() + np.abs(ve).max()
        assert np.abs(S @ ze - ve).max() <= (1e-12 if arm == "fp64" else 2e-3) * scale, e


@pytest.mark.parametrize("arm,n,N", [("fp64", 7, 4), ("fp64", 8, 4), ("fp64", 7, 5), ("mixed", 12, 5)])
def test_sweep_lists_in_every_form(arm, n, N):
    """Red rows S_rr z_r = v_r; black rows S_bb z_b = v_b - (S z_red)_b with the condensed operator."""
    from paper_1911_02366_gb300 import sc
    ctx = _system(arm, n, N, sc.SC_PC_RED_BLACK)
    K, _, _, nb = ctx.sc_sizes()
    v = np.random.default_rng(N).standard_normal(K * nb)
    z = _apply(ctx.sc_precond_apply, v)
    col = O.checkerboard(n)
    t = _apply(ctx.sc_condensed_matvec, np.where(np.repeat(col == 0, nb), z, 0.0))
    red, black = np.flatnonzero(col == 0), np.flatnonzero(col == 1)
    for e in (red[0], red[-1], black[0], black[-1]):
        S, sl = _schur_block(ctx, int(e), N), slice(e * nb, (e + 1) * nb)
        r = S @ z[sl] - v[sl] + (t[sl] if col[e] == 1 else 0.0)
        scale = np.abs(S).sum(axis=1).max() * np.abs(z[sl]).max() + np.abs(v[sl]).max() + np.abs(t[sl]).max()
        assert np.abs(r).max() <= (1e-12 if arm == "fp64" else 2e-3) * scale, (e, col[e])
