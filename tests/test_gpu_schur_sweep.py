"""The Schur-corrected sweep without tensor cores, and its dense red inverses at every order."""
import numpy as np
import pytest

import oracle as O
import oracle.sweep as SW
from gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _system(n, N, cfl=10.0, **cfg):
    from paper_1911_02366_gb300 import sc
    Q, dt, p, ctx = case(n, N, cfl=cfl, precision=sc.SC_PREC_MIXED, **cfg)
    ctx.sc_set_state(Q, Q)
    ctx.sc_assemble()
    ctx.sc_condense()
    return Q, dt, p, ctx


def _apply(ctx, v):
    z = torch.zeros(v.size, dtype=torch.float64, device="cuda")
    ctx.sc_precond_apply(torch.tensor(v, device="cuda"), z)
    return z.cpu().numpy()


@pytest.mark.parametrize("n,N", [(4, 2), (2, 3)])
def test_corrected_blocks_without_tensor_cores(n, N):
    """S_rr z_r = v_r and D_b z_b = v_b - sum_m S_bm z_m with the oracle's dense S and face-block Schur
    blocks D_b, to the backward error of the sweep with tensor cores (FP32 blocks and inverses)."""
    from paper_1911_02366_gb300 import sc
    Q, dt, p, ctx = _system(n, N, precond=sc.SC_PC_RB_SCHUR, tensor_cores=0)
    S = O.condensed_operator(O.jacobian(p, Q), n, N).dense_S()
    K = n ** 3
    nb = S.shape[0] // K
    D = SW.face_schur_blocks(S, n, N)
    v = np.random.default_rng(4).standard_normal(S.shape[0])
    z = _apply(ctx, v)
    col = O.checkerboard(n)
    t = S @ np.where(np.repeat(col == 0, nb), z, 0.0)
    scale = np.max(np.sum(np.abs(S), axis=1)) * np.max(np.abs(z)) + np.max(np.abs(v))
    for e in range(K):
        sl = slice(e * nb, (e + 1) * nb)
        M = D[e] if col[e] == 1 else S[sl, sl]
        r = M @ z[sl] - v[sl] + (t[sl] if col[e] == 1 else 0.0)
        assert np.max(np.abs(r)) <= (1e-4 if col[e] == 1 else 2e-5) * scale, (e, col[e])


def test_iterations_without_tensor_cores():
    """4^3 elements, N = 3, CFL-13 time step: 50 iterations with the plain sweep, 34 with the corrected one in
    the oracle's experiments, whatever multiplies the blocks."""
    from paper_1911_02366_gb300 import sc
    its = {}
    for pc in (sc.SC_PC_RED_BLACK, sc.SC_PC_RB_SCHUR):
        Q, dt, p, ctx = _system(4, 3, cfl=13.0, precond=pc, tensor_cores=0, rel_tol=1e-8, inner_tol=1e-4, max_refine=20)
        its[pc] = ctx.sc_solve(torch.zeros(Q.size, dtype=torch.float64, device="cuda"))["gmres_iters"]
    assert its[sc.SC_PC_RB_SCHUR] < 0.8 * its[sc.SC_PC_RED_BLACK], its


@pytest.mark.parametrize("tc", [0, 1])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 6])
def test_red_inverses_solve_the_element_schur_blocks(N, tc):
    """The red rows of one application, S_ee z_e = v_e with S_ee in FP64 from the assembled own block (n_b from
    130 to 1090: partial tiles of the inverse in both directions), as a backward error.  2e-3 as for
    block Jacobi with TF32 products; FP32 products alone leave a few 1e-6, here 1e-4."""
    from paper_1911_02366_gb300 import sc
    n = 2
    Q, dt, p, ctx = _system(n, N, precond=sc.SC_PC_RB_SCHUR, tensor_cores=tc)
    K, _, _, nb = ctx.sc_sizes()
    v = np.random.default_rng(N).standard_normal(K * nb)
    z = _apply(ctx, v)
    i = np.arange(N + 1)
    inner1 = (i > 0) & (i < N)
    inner = np.repeat((inner1[:, None, None] & inner1[None, :, None] & inner1[None, None, :]).reshape(-1), 5)
    col = O.checkerboard(n)
    for e in np.flatnonzero(col == 0)[[0, -1]]:
        A = ctx.sc_get_jacobian_block(int(e), int(e))
        S = A[np.ix_(~inner, ~inner)] - A[np.ix_(~inner, inner)] @ np.linalg.solve(A[np.ix_(inner, inner)],
                                                                                   A[np.ix_(inner, ~inner)])
        ze, ve = z[e * nb:(e + 1) * nb], v[e * nb:(e + 1) * nb]
        scale = np.abs(S).sum(axis=1).max() * np.abs(ze).max() + np.abs(ve).max()
        assert np.abs(S @ ze - ve).max() <= (2e-3 if tc else 1e-4) * scale, e


def test_measured_solves_are_those_with_factors():
    """The block-solve span of one application: the black elements' solve, not the product with the red
    inverses, which is another kernel."""
    from paper_1911_02366_gb300 import sc
    Q, dt, p, ctx = _system(4, 2, precond=sc.SC_PC_RB_SCHUR)
    K, _, _, nb = ctx.sc_sizes()
    ctx.sc_profile_kernel(sc.SC_KERNEL_LU_SOLVE)
    _apply(ctx, np.ones(K * nb))
    assert (ctx.sc_profile_read()[0], ctx.sc_profile_elements()) == (1, K // 2)
