"""Contexts of different orders used by host threads at the same time, each on its own stream: a
kernel's shared-memory limit belongs to the function, not to the caller's mesh."""
import threading

import numpy as np
import pytest

import sc_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(jobs):
    """Each job on a thread of its own, started together; the first exception is raised."""
    errors, gate = [], threading.Barrier(len(jobs))

    def body(job):
        gate.wait()
        try:
            job()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
    ts = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def _context(N, **cfg):
    from paper_1911_02366_gb300 import sc
    st = torch.cuda.Stream()
    n = 2
    Q, dt = I.tgv_state(n, N, cfl=2.0)
    ctx = sc.Context(stream=st.cuda_stream, **{"precision": sc.SC_PREC_MIXED, **cfg})
    ctx.sc_set_mesh(n, 2 * np.pi, N)
    torch.cuda.synchronize()
    ctx.sc_set_timestep(dt, 1)
    ctx.sc_set_state(Q, Q)
    return ctx, Q, st


def test_explicit_marches_of_different_orders():
    """Residual kernels: 67 KB of shared memory per CTA at order 6, 26 KB at order 2.  Same results as alone."""
    ctxs = [_context(N) for N in (2, 6, 3, 6)]
    alone = []
    for c, Q, _ in ctxs:
        c.sc_explicit_march(0.1, 3)
        alone.append(c.sc_get_state(np.zeros(Q.size)).copy())
        c.sc_set_state(Q, Q)

    def job(c, Q, want):
        for _ in range(150):
            c.sc_set_state(Q, Q)
            c.sc_explicit_march(0.1, 3)
        assert np.array_equal(c.sc_get_state(np.zeros(Q.size)), want)
    _run([lambda a=a, w=w: job(a[0], a[1], w) for a, w in zip(ctxs, alone)])


@pytest.mark.parametrize("tc", [0, 1])
def test_condensations_of_different_orders(tc):
    """Packing, panels, triangle inverses, couplings of the Schur-corrected sweep."""
    from paper_1911_02366_gb300 import sc
    ctxs = [_context(N, precond=pc, tensor_cores=tc) for N, pc in ((2, sc.SC_PC_RB_SCHUR), (6, sc.SC_PC_RB_SCHUR),
                                                                   (3, sc.SC_PC_BLOCK_JACOBI), (5, sc.SC_PC_BLOCK_JACOBI))]

    def job(c):
        for _ in range(40):
            c.sc_assemble()
            c.sc_condense()
    _run([lambda c=c: job(c) for c, _, _ in ctxs])
    for c, Q, _ in ctxs:
        assert c.sc_solve(np.zeros(Q.size))["rel_residual"] <= 1.0000001e-8


def test_long_restarts_beside_short_ones():
    """The Gram-Schmidt sweeps ask for more than 48 KB of shared memory from 171 vectors on.  Without a
    preconditioner the systems take more iterations than that in one cycle."""
    from paper_1911_02366_gb300 import sc
    ctxs = [_context(3, precision=sc.SC_PREC_FP64, precond=sc.SC_PC_NONE, gmres_restart=r, gmres_max_iters=600)
            for r in (400, 200)]
    its = [0, 0]

    def job(k):
        c, Q, _ = ctxs[k]
        for _ in range(4):
            c.sc_assemble()
            c.sc_condense()
            its[k] = c.sc_solve(np.zeros(Q.size), raise_on_not_converged=False)["gmres_iters"]
    _run([lambda k=k: job(k) for k in (0, 1)])
    assert min(its) > 171, its
