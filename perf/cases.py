"""Measured cases: the work a user of this package has it do, through its Python entry points.

Every system is the seeded Taylor-Green state of the repository's own workloads (Ma 0.1,
Re 1600, Sutherland, perturbed by 1e-3), with the time step of the CFL rule.  Solves run
to a relative residual of 1e-12: a march that has to reach the steady tolerance 1e-9 of the
implicit experiment needs its linear solves well below it, and there two correct solvers agree
in the digits that are compared.  Kinds:

  newton   set_state, assemble, condense, solve of one Newton system (Context)
  mixed    the same on one mesh whose elements have different orders (MixedContext)
  batch    five systems of orders 2..6 condensed together, then solved (Batch)
  rk       explicit low-storage RK3 steps (sc_explicit_march)
  direct   BDF1 steps with a frozen Jacobian and the dense LU of S or A (sc_implicit_march)
  infer    the correction network on every boundary node of a mesh (MLP.forward)
  train    the gradients of one batch of the network's training (MLP.forward, loss, backward)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1911_02366_gb300 import sc

MA, RE, PR, GAMMA, TS, DELTA = 0.1, 1600.0, 0.72, 1.4, 110.4 / 288.15, 0.05
SIDE = 2.0 * math.pi
REL_TOL = 1e-12
PRECONDS = {"bj": sc.SC_PC_BLOCK_JACOBI, "rb": sc.SC_PC_RED_BLACK, "rbs": sc.SC_PC_RB_SCHUR}


def newton(name, n, N, arm, pc, cfl, bdf=1, flux="roe_br1"):
    return {"name": name, "kind": "newton", "n": n, "N": N, "arm": arm, "pc": pc, "cfl": float(cfl), "bdf": bdf,
            "flux": flux}


def listed():
    return [
        # the smallest system of the tests: every call is launches and host round trips
        newton("newton_2x2x2_N2_fp64", 2, 2, "fp64", "bj", 10),
        # the 20,480-DOF mesh of the parity workload on the default arm (FP64, block Jacobi)
        newton("newton_4x4x4_N3_fp64", 4, 3, "fp64", "bj", 13),
        # the same mesh on the mixed arm with the benchmark's preconditioner, a BDF2 step
        newton("newton_4x4x4_N3_mixed_bdf2", 4, 3, "mixed", "rbs", 13, bdf=2),
        # the benchmark's workload: the largest system
        newton("newton_16x16x16_N4_mixed", 16, 4, "mixed", "rbs", 50),
        # an odd mesh of a high order (interior blocks of 320, face blocks of 760)
        newton("newton_9x9x9_N5_mixed", 9, 5, "mixed", "rbs", 30),
        # the highest order, with the Lax-Friedrichs / interior-penalty flux pair
        newton("newton_6x6x6_N6_mixed_lf_sipg", 6, 6, "mixed", "bj", 15, flux="lf_sipg"),
        # one mesh of uneven orders with mortar faces
        {"name": "mixedmesh_6x6x6_N2to6", "kind": "mixed", "n": 6, "cfl": 10.0},
        # five systems of uneven orders condensed in one batch
        {"name": "batch_5x5x5_N2to6", "kind": "batch", "n": 5, "cfl": 10.0},
        # an explicit march, the experiment's other time integrator
        {"name": "march_rk3_8x8x8_N4", "kind": "rk", "n": 8, "N": 4, "cfl": 0.15, "steps": 40},
        # frozen-Jacobian BDF1 steps through the dense LU of the condensed matrix
        {"name": "march_direct_3x3x3_N3_fp64", "kind": "direct", "n": 3, "N": 3, "arm": "fp64", "which": "S",
         "cfl": 10.0, "steps": 3},
        # the network over the boundary nodes of 1,024 elements of order 4
        {"name": "mlp_infer_100352", "kind": "infer", "samples": 100352},
        # one training batch of the benchmark's size
        {"name": "mlp_train_256", "kind": "train", "samples": 256},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["newton", "newton", "newton", "newton", "mixed", "batch", "rk", "direct", "infer", "train"])
    if kind == "newton":
        arm = rng.choice(["fp64", "mixed", "mixed"])
        N = rng.randint(2, 5 if arm == "fp64" else 6)
        dofs = _log_int(rng, 1080, 130000 if arm == "fp64" else 1500000)
        n = max(2, int(round((dofs / (5.0 * (N + 1) ** 3)) ** (1.0 / 3.0))))
        pc = rng.choice(["bj", "rb"] if arm == "fp64" else ["bj", "rb", "rbs", "rbs"])
        # time steps up to the benchmark's, whose CFL number is 50 at n N = 64
        cfl = round(max(4.0, rng.uniform(20.0, 50.0) * min(1.0, n * N / 64.0)), 2)
        c = newton("", n, N, arm, pc, cfl, bdf=rng.choice([1, 1, 2]), flux=rng.choice(["roe_br1", "roe_br1", "lf_sipg"]))
        del c["name"]
        return c
    if kind == "mixed":
        return {"kind": "mixed", "n": rng.randint(2, 6), "cfl": round(rng.uniform(4.0, 10.0), 2)}
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(2, 5), "cfl": round(rng.uniform(4.0, 10.0), 2)}
    if kind == "rk":
        N = rng.randint(2, 6)
        n = max(2, int(round((_log_int(rng, 1080, 1000000) / (5.0 * (N + 1) ** 3)) ** (1.0 / 3.0))))
        return {"kind": "rk", "n": n, "N": N, "cfl": round(rng.uniform(0.05, 0.15), 3), "steps": rng.randint(5, 40)}
    if kind == "direct":
        n, N = rng.choice([(2, 2), (3, 2), (2, 3), (4, 2), (3, 3)])
        arm = rng.choice(["fp64", "mixed"])
        return {"kind": "direct", "n": n, "N": N, "arm": arm, "which": rng.choice(["S", "S", "A"]) if n < 4 else "S",
                "cfl": round(rng.uniform(4.0, 8.0), 2), "steps": rng.randint(1, 3)}
    if kind == "infer":
        return {"kind": "infer", "samples": _log_int(rng, 200, 400000)}
    return {"kind": "train", "samples": _log_int(rng, 50, 1000)}


# ---- inputs ---------------------------------------------------------------------------------
def lobatto(N):
    """Gauss-Lobatto nodes, weights and differentiation matrix of order N."""
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(np.real(P.deriv().roots())), [1.0]])
    for _ in range(3):  # polish the roots of P_N'
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    x = 0.5 * (x - x[::-1])
    w = 2.0 / (N * (N + 1) * P(x) ** 2)
    b = np.array([1.0 / np.prod([x[j] - x[k] for k in range(N + 1) if k != j]) for j in range(N + 1)])
    D = np.zeros((N + 1, N + 1))
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = b[j] / b[i] / (x[i] - x[j])
        D[i, i] = -D[i].sum()
    return x, w, D


def _smooth(x, y, z):
    """The Taylor-Green state at the points, and its largest signal speed."""
    u, v = torch.sin(x) * torch.cos(y) * torch.cos(z), -torch.cos(x) * torch.sin(y) * torch.cos(z)
    p = 1.0 / (GAMMA * MA * MA) + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
    rho = GAMMA * MA * MA * p
    q = torch.stack([rho, rho * u, rho * v, torch.zeros_like(u), p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)], -1)
    return q, float((torch.sqrt(u * u + v * v) + torch.sqrt(GAMMA * p / rho)).max())


def _points(n, N):
    """Coordinates of every node, element by element, x fastest in elements and nodes."""
    x = torch.tensor(lobatto(N)[0], device="cuda")
    e = torch.arange(n, device="cuda", dtype=torch.float64)
    line = (SIDE / n) * (e[:, None] + 0.5 * (1.0 + x)[None, :])  # [element, node]
    p = N + 1
    shape = (n, n, n, p, p, p)  # ez, ey, ex, k, j, i
    X = line.view(1, 1, n, 1, 1, p).expand(shape).reshape(n ** 3, p ** 3)
    Y = line.view(1, n, 1, 1, p, 1).expand(shape).reshape(n ** 3, p ** 3)
    Z = line.view(n, 1, 1, p, 1, 1).expand(shape).reshape(n ** 3, p ** 3)
    return X, Y, Z


def _noise(q, gen):
    """Every value perturbed by 1e-3 of itself, and the momenta by 1e-3 of the free stream's (a developed
    flow has no component that is exactly zero, where the Lax-Friedrichs speed |u . n| has its kink)."""
    u = 2.0 * torch.rand(2, *q.shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0
    moving = torch.tensor([0.0, 1.0, 1.0, 1.0, 0.0], dtype=torch.float64, device="cuda")
    return q * (1.0 + 1e-3 * u[0]) + 1e-3 * u[1] * moving


def _state(n, N, cfl, seed):
    """Perturbed states (iterate, level s, level s - 1), flat, and the time step."""
    q, speed = _smooth(*_points(n, N))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    Q = _noise(q, gen)
    Qm = q + 0.9 * (Q - q)  # a slightly smoother earlier level
    return Q.reshape(-1).contiguous(), Q.reshape(-1).clone(), Qm.reshape(-1).contiguous(), cfl * (SIDE / n / N) / speed


def _config(arm, pc, flux="roe_br1"):
    lf, ip = flux == "lf_sipg", flux == "lf_sipg"
    return dict(precision=sc.SC_PREC_FP64 if arm == "fp64" else sc.SC_PREC_MIXED, Ma=MA, Re=RE, rel_tol=REL_TOL,
                precond=PRECONDS[pc], max_refine=20, adv_flux=sc.SC_FLUX_LF if lf else sc.SC_FLUX_ROE,
                visc_flux=sc.SC_VISC_SIPG if ip else sc.SC_VISC_BR1)


def _context(n, N, arm, pc, flux="roe_br1"):
    ctx = sc.Context(stream=torch.cuda.current_stream().cuda_stream, **_config(arm, pc, flux))
    ctx.sc_set_mesh(n, SIDE, N)
    return ctx


def _orders(n):
    return np.random.RandomState(1).randint(2, 7, n ** 3).astype(np.int32)


def _network(seed, samples):
    """Weights, biases, features and targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    W = torch.cat([(r(256, 128) * math.sqrt(2 / 128)).reshape(-1), (r(256, 256) * math.sqrt(2 / 256)).reshape(-1),
                   (r(25, 256) * 0.1 / 16).reshape(-1)])
    b = 0.01 * r(sc.MLP_NB)
    X = torch.zeros(samples, 128, device="cuda")
    X[:, :113] = r(samples, 113) / 5.0  # four unit-norm 5 x 5 blocks and 13 scalars; the rest is padding
    return W, b, X, 0.3 * r(samples, 25)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "newton":
        Q, Qs, Qm, dt = _state(case["n"], case["N"], case["cfl"], seed)
        ctx = _context(case["n"], case["N"], case["arm"], case["pc"], case["flux"])
        ctx.sc_set_timestep(dt, case["bdf"])
        return {"kind": kind, "ctx": ctx, "Q": Q, "Qs": Qs, "Qm": Qm if case["bdf"] == 2 else None,
                "B": torch.empty_like(Q), "dQ": torch.empty_like(Q)}
    if kind == "mixed":
        n, orders = case["n"], _orders(case["n"])
        qs, speed = {}, 0.0
        for N in np.unique(orders):
            qs[int(N)], s = _smooth(*_points(n, int(N)))
            speed = max(speed, s)
        q = torch.cat([qs[int(N)][e] for e, N in enumerate(orders)])
        Q = _noise(q, torch.Generator(device="cuda").manual_seed(seed)).reshape(-1).contiguous()
        ctx = sc.MixedContext(n, orders, SIDE, stream=torch.cuda.current_stream().cuda_stream, **_config("mixed", "bj"))
        return {"kind": kind, "ctx": ctx, "Q": Q, "dt": case["cfl"] * (SIDE / n / int(orders.max())) / speed,
                "R": torch.empty_like(Q), "dQ": torch.empty_like(Q)}
    if kind == "batch":
        systems = []
        for N in range(2, 7):
            Q, Qs, _, dt = _state(case["n"], N, case["cfl"], seed + 7919 * N)
            ctx = _context(case["n"], N, "mixed", "bj")
            ctx.sc_set_timestep(dt, 1)
            systems.append({"ctx": ctx, "Q": Q, "Qs": Qs, "dQ": torch.empty_like(Q)})
        return {"kind": kind, "systems": systems, "batch": sc.Batch([s["ctx"] for s in systems])}
    if kind == "rk":
        Q, _, _, _ = _state(case["n"], case["N"], case["cfl"], seed)
        ctx = sc.Context(stream=torch.cuda.current_stream().cuda_stream, **_config("mixed", "bj"))
        ctx.sc_set_mesh(case["n"], SIDE, case["N"])
        return {"kind": kind, "ctx": ctx, "Q": Q, "out": torch.empty_like(Q), "cfl": case["cfl"], "steps": case["steps"]}
    if kind == "direct":
        Q, _, _, dt = _state(case["n"], case["N"], case["cfl"], seed)
        ctx = _context(case["n"], case["N"], case["arm"], "bj")
        return {"kind": kind, "ctx": ctx, "Q": Q, "out": torch.empty_like(Q), "dt": dt, "steps": case["steps"],
                "which": case["which"]}
    n = case["samples"]
    W, b, X, T = _network(seed, n)
    net = sc.MLP(W.cpu().numpy(), b.cpu().numpy(), stream=torch.cuda.current_stream().cuda_stream)
    new = lambda *s: torch.empty(*s, device="cuda")  # noqa: E731
    st = {"kind": kind, "net": net, "X": X, "Y": new(n, 25)}
    if kind == "train":
        st |= {"T": T, "dY": new(n, 25), "cache": new(4, n, 256), "work": new(2, n, 256), "loss": new(1)}
    return st


def run(state):
    kind = state["kind"]
    if kind == "newton":
        ctx = state["ctx"]
        ctx.sc_set_state(state["Q"], state["Qs"], state["Qm"])
        ctx.sc_assemble()
        ctx.sc_get_rhs(state["B"])
        ctx.sc_condense()
        ctx.sc_solve(state["dQ"])
        return {"B": state["B"], "dQ": state["dQ"]}
    if kind == "mixed":
        ctx = state["ctx"]
        ctx.set_state(state["Q"], dt=state["dt"])
        ctx.residual(state["R"])
        ctx.condense()
        ctx.solve(state["dQ"])
        return {"R": state["R"], "dQ": state["dQ"]}
    if kind == "batch":
        for s in state["systems"]:
            s["ctx"].sc_set_state(s["Q"], s["Qs"])
            s["ctx"].sc_assemble()
        state["batch"].condense()
        for s in state["systems"]:
            s["ctx"].sc_solve(s["dQ"])
        return {"dQ": [s["dQ"] for s in state["systems"]]}
    if kind == "rk":
        ctx = state["ctx"]
        ctx.sc_set_state(state["Q"])
        res, dts, _ = ctx.sc_explicit_march(state["cfl"], state["steps"])
        return {"Q": ctx.sc_get_state(state["out"]), "residual": res, "dt": dts}
    if kind == "direct":
        ctx = state["ctx"]
        ctx.sc_set_state(state["Q"])
        res, _, _ = ctx.sc_implicit_march(state["dt"], state["steps"], direct=state["which"])
        return {"Q": ctx.sc_get_state(state["out"]), "residual": res}
    if kind == "infer":
        return {"Y": state["net"].forward(state["X"], state["Y"])}
    net = state["net"]
    for t in (net.gW, net.gb, state["loss"]):
        t.zero_()
    net.forward(state["X"], state["Y"], state["cache"])
    net.loss(state["Y"], state["T"], state["dY"], state["loss"])
    net.backward(state["X"], state["cache"], state["dY"], state["work"])
    return {"Y": state["Y"], "loss": state["loss"], "gW": net.gW, "gb": net.gb}


# ---- necessary work -------------------------------------------------------------------------
def _system_work(K, N, word, solve=True):
    """One system of K elements of order N: the states in, the update out and the element blocks'
    structural nonzeros once; the flops of the interior inverse, the Schur block and its LU."""
    nn, nin = (N + 1) ** 3, (N - 1) ** 3
    ni, nb = 5 * nin, 5 * (nn - nin)
    pairs = nn * (nn - N ** 3)  # node pairs sharing a GL index
    data = 8.0 * 5 * nn * 4 + word * 25.0 * (pairs + 6 * 5 * (N + 1) ** 2)
    flops = 2.0 * ni ** 3 + 2.0 * ni * ni * nb + 2.0 * nb * nb * ni + 2.0 / 3.0 * nb ** 3 + 4.0 * 25.0 * pairs
    return K * data, K * flops


def work(case):
    kind = case["kind"]
    if kind == "newton":
        b, f = _system_work(case["n"] ** 3, case["N"], 8.0 if case["arm"] == "fp64" else 4.0)
    elif kind in ("mixed", "batch"):
        K = case["n"] ** 3 / (5.0 if kind == "mixed" else 1.0)  # elements per order, on average
        parts = [_system_work(K, N, 4.0) for N in range(2, 7)]
        b, f = sum(x[0] for x in parts), sum(x[1] for x in parts)
    elif kind == "rk":
        dofs, p = 5.0 * case["n"] ** 3 * (case["N"] + 1) ** 3, case["N"] + 1
        b = 2.0 * 8.0 * dofs  # the state in and out
        f = case["steps"] * 3.0 * dofs * (12.0 * p + 120.0)  # lifting and divergence lines, point fluxes
    elif kind == "direct":
        K, N = case["n"] ** 3, case["N"]
        rows = 5.0 * K * ((N + 1) ** 3 - ((N - 1) ** 3 if case["which"] == "S" else 0))
        b = (8.0 if case["arm"] == "fp64" else 4.0) * rows * rows + 16.0 * 5 * K * (N + 1) ** 3
        f = 2.0 / 3.0 * rows ** 3 + case["steps"] * 2.0 * rows * rows
    else:
        s, params = float(case["samples"]), sc.MLP_NW + sc.MLP_NB
        b = 4.0 * s * (128 + 25) + (2.0 if kind == "infer" else 6.0) * params
        f = 2.0 * s * sc.MLP_NW * (1.0 if kind == "infer" else 3.0)
    return {"bytes": b, "flops": f}


# ---- the same results in 64 bits ------------------------------------------------------------
class _Operator:
    """The GL-DGSEM operator on a uniform periodic mesh in plain torch: states [..., n, n, n, p, p, p, 5]
    (elements z, y, x; nodes z, y, x), strong form."""

    def __init__(self, n, N, flux="roe_br1"):
        self.n, self.N, self.p, self.h = n, N, N + 1, SIDE / n
        _, w, D = lobatto(N)
        self.D = torch.tensor(D, device="cuda")
        self.w = torch.tensor(w, device="cuda")
        self.lf = self.ip = flux == "lf_sipg"
        self.sigma = (N + 1.0) ** 2 / (self.h * RE)

    def shape(self, q):
        return q.reshape(*q.shape[:-1], self.n, self.n, self.n, self.p, self.p, self.p, 5)

    @staticmethod
    def _ax(a):  # element and node axis of direction a (variables last)
        return -5 - a, -2 - a

    def line(self, q, a):
        ax = self._ax(a)[1]
        return torch.movedim(torch.matmul(torch.movedim(q, ax, -1), self.D.T), -1, ax)

    def face(self, q, a, side):
        return q.select(self._ax(a)[1], self.N if side > 0 else 0)

    def across(self, q, a, side):
        """The neighbour's values at the points of the face (a, side)."""
        f = q.select(self._ax(a)[1], 0 if side > 0 else self.N)
        return torch.roll(f, -1 if side > 0 else 1, self._ax(a)[0] + 1)

    def on_face(self, f, a, side):
        """Face values as a volume array, zero off the face."""
        ax = self._ax(a)[1]
        z = torch.zeros_like(f).unsqueeze(ax)
        rest = [z] * self.N
        return torch.cat(rest + [f.unsqueeze(ax)] if side > 0 else [f.unsqueeze(ax)] + rest, ax)

    def gradient(self, q, lifted):
        g = []
        for a in range(3):
            d = self.line(q, a)
            if lifted:
                for s in (-1, 1):
                    jump = self.across(q, a, s) - self.face(q, a, s)
                    d = d + self.on_face(0.5 * s / self.w[0] * jump, a, s)
            g.append(2.0 / self.h * d)
        return g

    @staticmethod
    def prim(q):
        r = q[..., 0]
        u = [q[..., 1 + i] / r for i in range(3)]
        kin = 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        return r, u, kin, (GAMMA - 1.0) * (q[..., 4] - r * kin)

    def inviscid(self, q, d):
        r, u, _, p = self.prim(q)
        f = [r * u[d]] + [r * u[d] * u[i] + (p if i == d else 0.0) for i in range(3)] + [(q[..., 4] + p) * u[d]]
        return torch.stack(f, -1)

    def viscous(self, q, g, d):
        r, u, kin, p = self.prim(q)
        du = [[(g[a][..., 1 + i] - u[i] * g[a][..., 0]) / r for i in range(3)] for a in range(3)]
        e = q[..., 4] / r - kin
        de = (g[d][..., 4] - q[..., 4] / r * g[d][..., 0]) / r - sum(u[i] * du[d][i] for i in range(3))
        T = GAMMA * (GAMMA - 1.0) * MA * MA * e
        mu = (1.0 + TS) * T * torch.sqrt(T) / (T + TS)
        div = du[0][0] + du[1][1] + du[2][2]
        tau = [mu * (du[d][i] + du[i][d] - (2.0 / 3.0 * div if i == d else 0.0)) for i in range(3)]
        heat = GAMMA / PR * mu * de
        f = [torch.zeros_like(r)] + tau + [sum(u[i] * tau[i] for i in range(3)) + heat]
        return torch.stack(f, -1) / RE

    def numerical(self, qa, qb, d, s):
        fa, fb = self.inviscid(qa, d), self.inviscid(qb, d)
        ra, ua, ka, pa = self.prim(qa)
        rb, ub, kb, pb = self.prim(qb)
        if self.lf:
            wa, wb = ua[d].abs() + torch.sqrt(GAMMA * pa / ra), ub[d].abs() + torch.sqrt(GAMMA * pb / rb)
            lam = torch.where(wa >= wb, wa, wb)
            return 0.5 * s * (fa + fb) - 0.5 * lam.unsqueeze(-1) * (qb - qa)
        sa, sb = torch.sqrt(ra), torch.sqrt(rb)
        u = [(sa * ua[i] + sb * ub[i]) / (sa + sb) for i in range(3)]
        H = (sa * (qa[..., 4] + pa) / ra + sb * (qb[..., 4] + pb) / rb) / (sa + sb)
        kin = 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        c = torch.sqrt((GAMMA - 1.0) * (H - kin))
        rho, un = sa * sb, s * u[d]
        dr, dp, dv = rb - ra, pb - pa, [ub[i] - ua[i] for i in range(3)]
        dun = s * dv[d]
        fix = lambda x: torch.where(x.abs() >= DELTA * c, x.abs(), (x * x + (DELTA * c) ** 2) / (2.0 * DELTA * c))  # noqa: E731
        am, ap = fix(un - c) * (dp - rho * c * dun) / (2 * c * c), fix(un + c) * (dp + rho * c * dun) / (2 * c * c)
        a0, ent = fix(un), dr - dp / (c * c)
        tang = [torch.zeros_like(c) if i == d else dv[i] for i in range(3)]
        mom = [(am + ap) * u[i] + a0 * (ent * u[i] + rho * tang[i]) + ((ap - am) * c * s if i == d else 0.0) for i in range(3)]
        en = (am + ap) * H + (ap - am) * c * un + a0 * (ent * kin + rho * sum(u[i] * tang[i] for i in range(3)))
        return 0.5 * s * (fa + fb) - 0.5 * torch.stack([am + ap + a0 * ent] + mom + [en], -1)

    def mass(self):
        w = self.w
        return (0.5 * self.h) ** 3 * (w[:, None, None] * w[None, :, None] * w[None, None, :]).unsqueeze(-1)

    def spatial(self, q):
        """M^-1 H(q) as an array like q."""
        g = self.gradient(q, True)
        gf = self.gradient(q, False) if self.ip else g
        r = torch.zeros_like(q)
        for d in range(3):
            F = self.inviscid(q, d) - self.viscous(q, g, d)
            r = r + self.line(F, d)
            for s in (-1, 1):
                qa, qb = self.face(q, d, s), self.across(q, d, s)
                fva = self.viscous(qa, [self.face(x, d, s) for x in gf], d)
                fvb = self.viscous(qb, [self.across(x, d, s) for x in gf], d)
                fh = self.numerical(qa, qb, d, s) - 0.5 * s * (fva + fvb)
                if self.ip:
                    fh = fh + self.sigma * (qa - qb)
                r = r + self.on_face((fh - s * self.face(F, d, s)) / self.w[0], d, s)
        return 2.0 / self.h * r

    def rhs(self, flat, hist, dt, c0):
        """B = -R(q) of a flat state."""
        q = self.shape(flat)
        r = self.spatial(q)
        if c0:
            r = r + c0 * (q - self.shape(hist)) / dt
        return -(self.mass() * r).reshape(flat.shape)

    def matrix(self, flat, dt, c0):
        """The dense Jacobian dR/dq, column by column in forward mode."""
        n, cols = flat.numel(), []
        f = lambda q: -self.rhs(q, flat, dt, c0)  # noqa: E731
        chunk = max(1, min(512, int(2e7 / n)))
        for j in range(0, n, chunk):
            k = min(chunk, n - j)
            e = torch.zeros(k, n, dtype=torch.float64, device="cuda")
            e[torch.arange(k), torch.arange(j, j + k)] = 1.0
            cols.append(torch.func.vmap(lambda t: torch.func.jvp(f, (flat,), (t,))[1])(e))
        return torch.cat(cols).T.contiguous()


DENSE_MOST = 21000  # unknowns of a dense 64-bit solve that stays well under 20 seconds


def _refined_solve(LU, A, b):
    x = torch.linalg.lu_solve(*LU, b.unsqueeze(1))
    return (x + torch.linalg.lu_solve(*LU, b.unsqueeze(1) - A @ x)).squeeze(1)


def _exact_update(op, Q, B, dt, c0):
    if Q.numel() > DENSE_MOST:
        return None
    A = op.matrix(Q, dt, c0)
    return _refined_solve(torch.linalg.lu_factor(A), A, B)


def _exact_rk(op, Q, cfl, steps):
    q, dx, res, dts = op.shape(Q).clone(), op.h / op.N, [], []
    dq = torch.zeros_like(q)
    for _ in range(steps):
        r, u, kin, p = op.prim(q)
        dt = cfl * dx / (torch.sqrt(2.0 * kin) + torch.sqrt(GAMMA * p / r)).max()
        dts.append(float(dt))
        for k, (a, b) in enumerate(((0.0, 1.0 / 3.0), (-5.0 / 9.0, 15.0 / 16.0), (-153.0 / 128.0, 8.0 / 15.0))):
            rate = -op.spatial(q)
            if k == 0:
                res.append(float(rate.abs().max()))
            dq = a * dq + dt * rate
            q = q + b * dq
    res.append(float(op.spatial(q).abs().max()))
    return {"Q": q.reshape(-1), "residual": np.array(res), "dt": np.array(dts)}


def _layers(W):
    return W[:32768].view(256, 128), W[32768:98304].view(256, 256), W[98304:].view(25, 256)


def exact(case, seed):
    kind = case["kind"]
    if kind == "newton":
        Q, Qs, Qm, dt = _state(case["n"], case["N"], case["cfl"], seed)
        op = _Operator(case["n"], case["N"], case["flux"])
        c0, hist = (1.5, (4.0 * Qs - Qm) / 3.0) if case["bdf"] == 2 else (1.0, Qs)
        B = op.rhs(Q, hist, dt, c0)
        return {"B": B, "dQ": _exact_update(op, Q, B, dt, c0)}
    if kind == "batch":  # the order-2 system fits a dense solve
        out = []
        for N in range(2, 7):
            Q, Qs, _, dt = _state(case["n"], N, case["cfl"], seed + 7919 * N)
            op = _Operator(case["n"], N)
            small = Q.numel() <= (DENSE_MOST if N == 2 else 5000)
            out.append(_exact_update(op, Q, op.rhs(Q, Qs, dt, 1.0), dt, 1.0) if small else None)
        return {"dQ": out}
    if kind == "mixed":
        return None  # tens of thousands of unknowns coupled through mortars: no dense solve in 20 s
    if kind == "rk":
        Q, _, _, _ = _state(case["n"], case["N"], case["cfl"], seed)
        return _exact_rk(_Operator(case["n"], case["N"]), Q, case["cfl"], case["steps"])
    if kind == "direct":
        Q, _, _, dt = _state(case["n"], case["N"], case["cfl"], seed)
        op = _Operator(case["n"], case["N"])
        A = op.matrix(Q, dt, 1.0)
        LU, res = torch.linalg.lu_factor(A), []
        for _ in range(case["steps"]):
            res.append(float(op.spatial(op.shape(Q)).abs().max()))
            Q = Q + _refined_solve(LU, A, op.rhs(Q, Q, dt, 0.0))
        res.append(float(op.spatial(op.shape(Q)).abs().max()))
        return {"Q": Q, "residual": np.array(res)}
    W, b, X, T = (t.double() for t in _network(seed, case["samples"]))
    W = W.float().to(torch.bfloat16).double().requires_grad_(kind == "train")  # the weights are used in BF16
    b.requires_grad_(kind == "train")
    W1, W2, W3 = _layers(W)
    h = torch.relu(torch.relu(X @ W1.T + b[:256]) @ W2.T + b[256:512])
    Y = h @ W3.T + b[512:]
    if kind == "infer":
        return {"Y": Y}
    loss = (((Y - T) ** 2).sum(1) / ((T ** 2).sum(1) + 1e-12)).mean()
    gW, gb = torch.autograd.grad(loss, [W, b])
    return {"Y": Y.detach(), "loss": loss.detach().reshape(1), "gW": gW, "gb": gb}
