"""What the framework is timed on: batches of multi-agent trajectory QPs solved, differentiated and
re-linearized through the public entry points (Solver, TADMMFunction).

The instances are of the kinds that instances/generator.py draws (a crossing, a ring, mixed boxes of agents
that swap places, a 3D swarm, boxes with a tracking loss), with the same model, costs, bounds and separations.
They are drawn here for a whole batch at a time, because inputs are made often: the constant-velocity guess of
a scenario is scaled back until every pair keeps 1.1 d_min along the whole line, which makes it feasible.
"""
import math

import numpy as np
import torch

import paper_2602_15838_gb300 as tg
from instances import Batch, double_integrator

DT = 0.1


# ----------------------------------------------------------------------------- the cases
def listed():
    return [
        # One crossing of two agents, the smallest problem anybody solves: a single call's latency.
        dict(name="crossing_2", kind="crossing", scen=1, nmin=2, nmax=2, tmin=20, tmax=20, iters=500),
        # One ring of fourteen agents that swap sides, the usual benchmark of the method, in the mode
        # for single scenarios (phase kernels repeated on the device).
        dict(name="ring_14_graph", kind="ring", scen=1, nmin=14, nmax=14, tmin=20, tmax=20, iters=300, mode="graph"),
        # Receding horizon: new data of a few hundred scenarios from the host each cycle, some iterations, the
        # answer back to the host.  Launch shape left to the library, as a first program has it.
        dict(name="receding_256", kind="mixed", run="cycle", scen=256, nmin=2, nmax=32, tmin=20, tmax=40, iters=30),
        # The throughput workload: thousands of ragged scenarios to the tolerance or 500 iterations, with
        # the launch shape that the autotuner keeps.
        dict(name="mixed_4096", kind="mixed", scen=4096, nmin=2, nmax=32, tmin=20, tmax=40, iters=500, tune=True),
        # The same kind of batch in float32, as used where 1e-4 is enough.
        dict(name="mixed_1024_f32", kind="mixed", scen=1024, nmin=2, nmax=32, tmin=20, tmax=40, iters=200, prec=32,
             tune=True),
        # Penalty balancing with over-relaxation, the options that make most scenarios converge.
        dict(name="balanced_relaxed_512", kind="mixed", scen=512, nmin=2, nmax=32, tmin=20, tmax=40, iters=150,
             adapt=True, relax=1.6),
        # Agents of unlike mass and damping, coupled by a communication graph (four links each) and not all to all.
        dict(name="unlike_linked_256", kind="mixed", scen=256, nmin=5, nmax=32, tmin=20, tmax=40, iters=100,
             unlike=True, links=2),
        # One large 3D swarm, all pairs coupled, in the mode for scenarios too large for one block.
        dict(name="swarm3d_512_graph", kind="swarm", scen=1, nmin=512, nmax=512, tmin=40, tmax=40, iters=20,
             mode="graph"),
        # Many small 3D swarms with ragged horizons in the batched mode.
        dict(name="swarms3d_200", kind="swarm", scen=200, nmin=3, nmax=25, tmin=20, tmax=40, iters=60),
        # A training step through the solver: solve, states at the active set, gradients of a tracking loss
        # with respect to the cost weights and the goals.
        dict(name="train_128x6", kind="tracking", run="train", scen=128, nmin=6, nmax=6, tmin=30, tmax=30, iters=400,
             adapt=True),
        # Refinement of a solve's active set on the centralized QP, then the gradients there.
        dict(name="polish_64x16", kind="tracking", run="polish", scen=64, nmin=16, nmax=16, tmin=30, tmax=30, iters=400,
             adapt=True, rounds=12),
        # The loop that linearizes the collision constraint again around each solution.
        dict(name="relinearize_96", kind="mixed", run="sqp", scen=96, nmin=2, nmax=16, tmin=20, tmax=30, iters=150,
             adapt=True, rounds=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["single", "single_graph", "mixed", "mixed", "mixed", "cycle", "options", "unlike", "swarm",
                       "swarms", "train", "polish", "sqp"])
    t0 = rng.randint(8, 40)
    t1 = rng.randint(t0, 40)
    prec = rng.choice([64, 64, 64, 32])
    if what == "single":
        n = rng.randint(2, 32)
        return dict(kind=rng.choice(["ring", "mixed"]), scen=1, nmin=n, nmax=n, tmin=t1, tmax=t1,
                    iters=_log(rng, 5, 300), prec=prec)
    if what == "single_graph":
        n = rng.randint(2, 40)
        return dict(kind=rng.choice(["ring", "mixed"]), scen=1, nmin=n, nmax=n, tmin=t1, tmax=t1,
                    iters=_log(rng, 5, 300), mode="graph", prec=prec)
    if what == "mixed":
        n0 = rng.randint(1, 16)
        return dict(kind="mixed", scen=_log(rng, 16, 3000), nmin=n0, nmax=rng.randint(n0 + 1, 32), tmin=t0, tmax=t1,
                    iters=_log(rng, 20, 400), prec=prec, tune=rng.random() < 0.5)
    if what == "cycle":
        return dict(kind="mixed", run="cycle", scen=_log(rng, 1, 1000), nmin=2, nmax=rng.randint(3, 32), tmin=t0, tmax=t1,
                    iters=_log(rng, 5, 60), prec=prec)
    if what == "options":
        return dict(kind="mixed", scen=_log(rng, 32, 1000), nmin=2, nmax=rng.randint(3, 32), tmin=t0, tmax=t1,
                    iters=_log(rng, 30, 200), adapt=rng.random() < 0.7, relax=rng.choice([1.0, 1.3, 1.6]))
    if what == "unlike":
        return dict(kind="mixed", scen=_log(rng, 16, 500), nmin=4, nmax=rng.randint(6, 32), tmin=t0, tmax=t1,
                    iters=_log(rng, 20, 120), unlike=rng.random() < 0.6, links=rng.choice([0, 1, 2, 4]))
    if what == "swarm":
        n = _log(rng, 40, 400)
        return dict(kind="swarm", scen=1, nmin=n, nmax=n, tmin=t1, tmax=t1, iters=_log(rng, 5, 30), mode="graph")
    if what == "swarms":
        return dict(kind="swarm", scen=_log(rng, 8, 300), nmin=2, nmax=rng.randint(4, 28), tmin=t0, tmax=t1,
                    iters=_log(rng, 20, 80), prec=prec)
    if what in ("train", "polish"):
        n = rng.randint(3, 8) if what == "train" else rng.randint(4, 20)
        c = dict(kind="tracking", run=what, scen=_log(rng, 4, 64), nmin=n, nmax=n, tmin=t1, tmax=t1,
                 iters=_log(rng, 100, 400), adapt=True)
        return c if what == "train" else dict(c, rounds=rng.randint(3, 10))
    return dict(kind="mixed", run="sqp", scen=_log(rng, 8, 128), nmin=2, nmax=rng.randint(4, 20), tmin=t0, tmax=t1,
                iters=_log(rng, 40, 150), adapt=rng.random() < 0.5, rounds=rng.randint(2, 4))


# ----------------------------------------------------------------------------- instances
def _starts(rng, N, dp, lo, hi, sep):
    """[scen, max N, dp] points, the first N[s] of a scenario pairwise at least `sep` apart."""
    S, n = len(N), int(N.max())
    pts = np.full((S, n, dp), 1e9)
    for k in range(n):
        left = np.flatnonzero(N > k)
        while len(left):
            c = rng.uniform(lo, hi, (len(left), 6, dp))
            if k:
                d = ((c[:, :, None] - pts[left, None, :k]) ** 2).sum(-1).min(-1)
                ok = d >= sep * sep
            else:
                ok = np.ones(c.shape[:2], bool)
            good = ok.any(1)
            pts[left[good], k] = c[good, ok[good].argmax(1)]
            left = left[~good]
    return pts


def _points(case, rng, N):
    """Starts and goals [scen, max N, dp] of the case's kind."""
    S, n = len(N), int(N.max())
    if case["kind"] in ("crossing", "ring"):
        sigma = 0.05 if case["kind"] == "crossing" else 0.1
        radius = 5.0 * max(1.0, n / 20.0)
        phi = 2.0 * math.pi * np.arange(n) / n
        ring = radius * np.stack([np.cos(phi), np.sin(phi)], axis=1)
        return (ring + sigma * rng.standard_normal((S, n, 2)), -ring + sigma * rng.standard_normal((S, n, 2)))
    if case["kind"] == "swarm":
        side = 20.0 if n > 64 else 8.0
        s = _starts(rng, N, 3, -side, side, 1.0)
        return s, -s
    box = 5.0 * max(1.0, math.sqrt(n / 32.0))
    s = _starts(rng, N, 2, -box, box, 0.8)
    key = np.where(np.arange(n)[None] < N[:, None], rng.random((S, n)), 2.0)
    return s, np.take_along_axis(s, np.argsort(key, axis=1)[:, :, None], axis=1)


def _batch(case, seed):
    rng = np.random.default_rng([20260215, int(seed)])
    S = int(case["scen"])
    dp = 3 if case["kind"] == "swarm" else 2
    nx, nu = 2 * dp, dp
    sizes = np.random.default_rng([S, case["nmin"], case["nmax"], case["tmin"], case["tmax"]])
    N = sizes.integers(case["nmin"], case["nmax"] + 1, S)   # a program's batch keeps its sizes, its data changes
    T = sizes.integers(case["tmin"], case["tmax"] + 1, S)
    d = 0.4 if case["kind"] in ("mixed", "tracking") else 0.5
    rho, umax = (2.0, 2.0) if dp == 3 else (1.0, 1.0)
    s, g = _points(case, rng, N)
    v = g - s
    # largest c in {1, 1/2, ..., 2^-20, 0} whose lines s + t v, t in [0, c], keep 1.1 d_min between all pairs
    n = int(N.max())
    c = np.zeros(S)
    iu, ju = np.triu_indices(n, 1)
    have = ju[None] < N[:, None]
    ds, dv = s[:, iu] - s[:, ju], v[:, iu] - v[:, ju]
    if len(iu):
        ss, sv, vv = (ds * ds).sum(-1), (ds * dv).sum(-1), (dv * dv).sum(-1)
        ss[~have] = 1e9
        best = -sv / np.maximum(vv, 1e-30)
        open_ = np.ones(S, bool)
        for k in range(21):
            cand = 2.0 ** -k
            t = np.clip(best[open_], 0.0, cand)
            near = (ss[open_] + t * (2.0 * sv[open_] + t * vv[open_])).min(1)
            hit = np.flatnonzero(open_)[near >= (1.1 * d) ** 2]
            c[hit] = cand
            open_[hit] = False
            if not open_.any():
                break
    else:
        c[:] = 1.0
    A, B = double_integrator(dp, DT)
    na, nas, nps = int(N.sum()), int((N * T).sum()), int((N * (N - 1) // 2 * T).sum())
    x_init, x_ref = np.empty((na, nx)), np.zeros((na, nx))
    a, w0 = np.empty((nps, dp)), np.empty((nas, dp))
    ao = wo = po = 0
    for k in range(S):
        Nk, Tk = int(N[k]), int(T[k])
        sk, vk = s[k, :Nk], c[k] * v[k, :Nk]
        x_init[ao:ao + Nk, :dp], x_init[ao:ao + Nk, dp:] = sk, vk / (Tk * DT)
        x_ref[ao:ao + Nk, :dp] = g[k, :Nk]
        tt = (np.arange(1, Tk + 1) / Tk)[:, None]
        line = sk[:, None] + tt * vk[:, None]
        w0[wo:wo + Nk * Tk] = line.reshape(-1, dp)
        Pk = Nk * (Nk - 1) // 2
        if Pk:
            i, j = np.triu_indices(Nk, 1)
            df = (line[i] - line[j]).reshape(-1, dp)
            nr = df[:, 0] * df[:, 0]
            for r in range(1, dp):
                nr += df[:, r] * df[:, r]
            np.divide(df, np.sqrt(nr)[:, None], out=a[po:po + Pk * Tk])
        ao, wo, po = ao + Nk, wo + Nk * Tk, po + Pk * Tk
    q = np.concatenate([np.full(dp, 1.0), np.full(dp, 0.1)])
    b = Batch(nx=nx, nu=nu, dp=dp, N=N.astype(np.int32), T=T.astype(np.int32), A=A, B=B, umin=np.full(nu, -umax),
              umax=np.full(nu, umax), Qd=np.tile(q, (na, 1)), Rd=np.full((na, nu), 0.1), Qfd=np.tile(10.0 * q, (na, 1)),
              x_init=x_init, x_ref=x_ref, a=a, w0=w0, d_min=np.full(S, d), rho=np.full(S, rho))
    if case["kind"] == "tracking":
        b.targets = rng.uniform(-5.0, 5.0, (nas, dp))
    if case.get("links"):
        _keep_links(b, int(case["links"]))
    if case.get("unlike"):
        # x' = x + dt v + dt^2 / 2m u, v' = (1 - c dt) v + dt / m u, per agent
        damp, mass = rng.uniform(0.0, 0.5, na), rng.uniform(0.8, 1.25, na)
        b.A_agent, b.B_agent = np.tile(A, (na, 1, 1)), B[None] / mass[:, None, None]
        b.A_agent[:, range(dp, nx), range(dp, nx)] = (1.0 - damp * DT)[:, None]
    return b.contiguous()


def _keep_links(b, k):
    """Couples each agent to the k after it around its scenario only (listed pairs, a subset of all)."""
    counts, lists, rows = [], [], []
    po = b.pairstep_off
    for s in range(b.n_scen):
        N, T = int(b.N[s]), int(b.T[s])
        i, j = np.triu_indices(N, 1)
        keep = np.minimum(j - i, N - (j - i)) <= k
        lists.append(np.stack([i[keep], j[keep]], axis=1))
        counts.append(int(keep.sum()))
        rows.append(b.a[po[s]:po[s + 1]].reshape(len(i), T, b.dp)[keep].reshape(-1, b.dp))
    b.a = np.concatenate(rows)
    b.pair_count, b.pair_ij = np.asarray(counts, np.int32), np.concatenate(lists).astype(np.int32)


# ----------------------------------------------------------------------------- prepare and run
def _solver(case, batch):
    kw = dict(precision=int(case.get("prec", 64)), mode=case.get("mode", "batched"), relax=float(case.get("relax", 1.0)))
    if case.get("adapt"):
        kw["adapt"] = (10, 10.0, 2.0)
    s = tg.Solver(batch, **kw)
    if case.get("tune"):
        s.autotune(probe_iter=8)
    return s


def prepare(case, seed):
    batch = _batch(case, seed)
    state = dict(case=case, solver=_solver(case, batch), tol=1e-4, iters=int(case["iters"]))
    how = case.get("run")
    if how == "cycle":
        state["batch"] = batch
    if how == "train":
        state["tol"] = 1e-6
        p = lambda v: torch.tensor(v, device="cuda", requires_grad=True)  # noqa: E731
        state.update(Q=p(batch.Qd), R=p(batch.Rd), goal=p(batch.x_ref), targets=torch.tensor(batch.targets, device="cuda"))
    if how == "polish":
        state["solver"].solve(1e-6, state["iters"])
        rng = np.random.default_rng([7, int(seed)])
        state["grad"] = torch.tensor(rng.standard_normal(state["solver"].sizes["X"]), device="cuda")
    return state


def run(state):
    case, s, tol, iters = state["case"], state["solver"], state["tol"], state["iters"]
    how = case.get("run")
    if how == "cycle":
        s.update(state["batch"])
        s.solve(tol, iters)
        return s.solution()
    if how == "train":
        Q, R, goal = state["Q"], state["R"], state["goal"]
        Q.grad = R.grad = goal.grad = None
        X = tg.TADMMFunction.apply(Q, R, goal, s, tol, iters)
        S, N, T = case["scen"], case["nmax"], case["tmax"]
        pos = X.view(S, N, T + 1, 4)[:, :, 1:, :2].reshape(-1, 2)
        loss = ((pos - state["targets"]) ** 2).sum()
        loss.backward()
        return dict(X=X.detach(), loss=loss.detach(), gQ=Q.grad, gR=R.grad, gGoal=goal.grad)
    if how == "polish":
        p = s.polish(1e-9, int(case["rounds"]))
        return dict(polish=p, grads=s.backward(state["grad"]))
    if how == "sqp":
        r = s.sqp(tol, iters, max_outer=int(case["rounds"]))
        return dict(loop=r, sol=s.solution(device=True))
    s.solve(tol, iters)
    return s.solution(device=True)


def work(case):
    dp = 3 if case["kind"] == "swarm" else 2
    n, t = (case["nmin"] + case["nmax"]) / 2, (case["tmin"] + case["tmax"]) / 2
    var = ((case["nmax"] - case["nmin"] + 1) ** 2 - 1) / 12
    pairs = (n * n + var - n) / 2
    if case.get("links"):
        pairs = min(pairs, n * case["links"])
    steps, psteps = case["scen"] * n * t, case["scen"] * pairs * t
    # per iteration: one pass backward and forward over each agent's stages (two states and one input for each
    # axis: 6 + 5 products and sums at two operations), and the projection of each pair-step with its two sums
    iters = 5 if case["kind"] == "crossing" else case["iters"]
    flops = iters * (steps * dp * 22 + psteps * (8 * dp + 4))
    size = 8 * (steps * dp + psteps * dp + case["scen"] * n * (8 * dp + dp))          # w0, a and the agents' rows
    size += steps * (8 * 2 * dp + 8 * dp + dp) + 8 * psteps                              # X, U, W and theta
    how = case.get("run")
    if how == "sqp":
        flops *= case["rounds"]
    if how == "train":
        flops += 2 * steps * dp * 22 * 2
    if how == "polish":
        flops = case["rounds"] * steps * dp * 22
    return dict(bytes=int(size), flops=int(flops))


# ----------------------------------------------------------------------------- the same in plain 64 bits
class _Plain:
    """The ADMM of a batch in its literal form (consensus copies w and scaled duals y per pair and side), every
    agent's QP condensed to its inputs and solved at its optimum, for all agents at once on padded horizons."""

    def __init__(self, b, case):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        f = lambda v: torch.tensor(np.asarray(v), dtype=torch.float64, device=dev)  # noqa: E731
        self.b, self.dev, self.dp, self.nx, self.nu = b, dev, b.dp, b.nx, b.nu
        N, T = b.N.astype(np.int64), b.T.astype(np.int64)
        self.Tm = Tm = int(T.max())
        S, na, dp, nx, nu = len(N), int(N.sum()), b.dp, b.nx, b.nu
        self.na = na
        asc = np.repeat(np.arange(S), N)
        off = np.concatenate([[0], np.cumsum(N)])
        pij = [b.pairs_of(k) + off[k] for k in range(S)]
        psc = np.repeat(np.arange(S), [len(p) for p in pij])
        pij = np.concatenate(pij) if len(pij) else np.zeros((0, 2), np.int64)
        i64 = lambda v: torch.tensor(np.asarray(v, dtype=np.int64), device=dev)  # noqa: E731
        self.asc, self.psc, self.pi, self.pj = i64(asc), i64(psc), i64(pij[:, 0]), i64(pij[:, 1])
        self.Ta, self.Tp = i64(T[asc]), i64(T[psc])
        tt = torch.arange(1, Tm + 1, device=dev)
        self.am, self.pm = tt[None] <= self.Ta[:, None], tt[None] <= self.Tp[:, None]
        self.a = torch.zeros(len(pij), Tm, dp, dtype=torch.float64, device=dev)
        self.a[self.pm] = f(b.a).reshape(-1, dp)
        self.w0 = torch.zeros(na, Tm, dp, dtype=torch.float64, device=dev)
        self.w0[self.am] = f(b.w0)
        self.d, self.rho = f(b.d_min), f(b.rho)
        self.nc = torch.zeros(na, dtype=torch.float64, device=dev)
        one = torch.ones(len(pij), dtype=torch.float64, device=dev)
        self.nc.index_add_(0, self.pi, one).index_add_(0, self.pj, one)
        A = f(b.A_agent) if b.A_agent is not None else f(b.A)[None]
        B = f(b.B_agent) if b.B_agent is not None else f(b.B)[None]
        M = A.shape[0]
        self.Phi = torch.zeros(M, Tm, nx, nx, dtype=torch.float64, device=dev)
        self.Gam = torch.zeros(M, Tm, nx, Tm, nu, dtype=torch.float64, device=dev)
        P, G = torch.eye(nx, dtype=torch.float64, device=dev).expand(M, nx, nx), self.Gam.new_zeros(M, nx, Tm, nu)
        for t in range(Tm):
            P = A @ P
            G = (A @ G.reshape(M, nx, -1)).reshape(M, nx, Tm, nu)
            G[:, :, t] = B
            self.Phi[:, t], self.Gam[:, t] = P, G
        self.q(f(b.Qd), f(b.Rd), f(b.Qfd), f(b.x_ref))
        self.x0 = f(b.x_init)
        self.lo, self.hi = f(b.umin).repeat(Tm), f(b.umax).repeat(Tm)

    def q(self, Qd, Rd, Qfd, ref):
        last = torch.arange(1, self.Tm + 1, device=self.dev)[None] == self.Ta[:, None]
        self.Q2 = 2.0 * torch.where(last[..., None], Qfd[:, None], Qd[:, None]) * self.am[..., None]
        self.R2 = torch.where(self.am[..., None], 2.0 * Rd[:, None], torch.ones_like(Rd)[:, None]).reshape(self.na, -1)
        self.ref = ref

    def hessian(self, rnc):
        """Condensed Hessian with rnc [agents] added to the positions' weights, and those weights."""
        W = self.Q2.clone()
        W[:, :, :self.dp] = W[:, :, :self.dp] + rnc[:, None, None] * self.am[..., None]
        G = self.Gam.reshape(self.Gam.shape[0], self.Tm * self.nx, -1)
        H = G.transpose(1, 2) @ (W.reshape(self.na, -1, 1) * G)
        return H + torch.diag_embed(self.R2), W

    def states(self, u):
        G = self.Gam.reshape(self.Gam.shape[0], self.Tm * self.nx, -1)
        X = (G @ u[..., None]).reshape(self.na, self.Tm, self.nx)
        return X + (self.Phi @ self.x0[:, None, :, None])[..., 0]

    def free(self):
        G = self.Gam.reshape(self.Gam.shape[0], self.Tm * self.nx, -1)
        return G, (self.Phi @ self.x0[:, None, :, None])[..., 0]

    def box(self, H, f, u, side):
        """Box QPs by the primal active set from feasible inputs and their working set (-1, 0, 1)."""
        u, side = u.clone(), side.clone()
        todo = torch.arange(self.na, device=self.dev)
        for _ in range(2000):
            Ht, ft, ut, st = H[todo], f[todo], u[todo], side[todo]
            held = st != 0
            rhs = torch.where(held, ut, -ft - (Ht @ (ut * held)[..., None])[..., 0])
            Hm = Ht * (~held)[:, :, None] * (~held)[:, None, :] + torch.diag_embed(held.to(H.dtype))
            full = torch.where(held, ut, torch.cholesky_solve(rhs[..., None], torch.linalg.cholesky(Hm))[..., 0])
            p = full - ut
            room = torch.where(p < 0, ut - self.lo, self.hi - ut).clamp_min(0.0)
            ratio = torch.where((p == 0) | held, torch.inf, room / p.abs())
            alpha, at = ratio.min(1)
            stop = alpha < 1.0
            new = torch.where(stop[:, None], ut + alpha.clamp_max(1.0)[:, None] * p, full)
            row = torch.arange(len(todo), device=self.dev)
            to = torch.where(p[row, at] < 0, -1, 1)
            new[row[stop], at[stop]] = torch.where(to < 0, self.lo[at], self.hi[at])[stop]
            g = (Ht @ full[..., None])[..., 0] + ft
            mu = torch.where(held, -st * g, torch.inf)
            worst, drop = mu.min(1)
            size = torch.where(held, g.abs(), 0.0).amax(1).clamp_min(1.0)
            leave = ~stop & (worst < -1e-12 * size)
            st[row[stop], at[stop]] = to[stop]
            st[row[leave], drop[leave]] = 0
            u[todo], side[todo] = new, st
            todo = todo[stop | leave]
            if not len(todo):
                return u, side
        raise ArithmeticError("a box QP did not come to its optimum")

    def solve(self, tol, iters, adapt=None, relax=1.0):
        S, dp = len(self.b.N), self.dp
        big = lambda v, idx: torch.zeros(S, dtype=torch.float64, device=self.dev).scatter_reduce_(0, idx, v, "amax")  # noqa: E731
        act = torch.ones(S, dtype=torch.bool, device=self.dev)
        rho = self.rho.clone()
        wi, wj = self.w0[self.pi], self.w0[self.pj]
        yi, yj = torch.zeros_like(wi), torch.zeros_like(wj)
        u = torch.zeros(self.na, self.Tm * self.nu, dtype=torch.float64, device=self.dev)
        side = torch.zeros(u.shape, dtype=torch.int64, device=self.dev)
        X = torch.zeros(self.na, self.Tm, self.nx, dtype=torch.float64, device=self.dev)
        theta = torch.zeros(len(self.pi), self.Tm, dtype=torch.float64, device=self.dev)
        res = torch.zeros(S, 2, dtype=torch.float64, device=self.dev)
        G, free = self.free()
        H, W = self.hessian(rho[self.asc] * self.nc)
        for k in range(iters):
            h = torch.zeros(self.na, self.Tm, dp, dtype=torch.float64, device=self.dev)
            h.index_add_(0, self.pi, wi - yi).index_add_(0, self.pj, wj - yj)
            lin = -self.Q2 * self.ref[:, None]
            lin[:, :, :dp] -= rho[self.asc][:, None, None] * h * self.am[..., None]
            f = (G.transpose(1, 2) @ (W * free + lin).reshape(self.na, -1, 1))[..., 0]
            if k == 0:  # the unconstrained optimum, cut to the box
                v = torch.cholesky_solve(-f[..., None], torch.linalg.cholesky(H))[..., 0]
                sn = torch.where(v < self.lo, -1, torch.where(v > self.hi, 1, 0))
                un = torch.maximum(torch.minimum(v, self.hi), self.lo)
            un, sn = self.box(H, f, un, sn)
            ga = act[self.asc]
            u, side = torch.where(ga[:, None], un, u), torch.where(ga[:, None], sn, side)
            X = torch.where(ga[:, None, None], self.states(u), X)
            p = X[:, :, :dp]
            pi, pj = p[self.pi], p[self.pj]
            vi, vj = relax * pi + (1.0 - relax) * wi, relax * pj + (1.0 - relax) * wj
            th = 0.5 * (self.d[self.psc][:, None] - (self.a * ((vi + yi) - (vj + yj))).sum(-1))
            th = th.clamp_min(0.0) * self.pm
            ni, nj = vi + yi + th[..., None] * self.a, vj + yj - th[..., None] * self.a
            m = self.pm[..., None]
            gp = act[self.psc][:, None]
            top = lambda e: (e.abs() * m).amax((1, 2)) if len(self.pi) else self.d.new_zeros(0)  # noqa: E731
            r = big(torch.maximum(top(pi - ni), top(pj - nj)), self.psc)
            s = rho * big(torch.maximum(top(ni - wi), top(nj - wj)), self.psc)
            yi = torch.where(gp[..., None], vi + yi - ni, yi)
            yj = torch.where(gp[..., None], vj + yj - nj, yj)
            wi, wj = torch.where(gp[..., None], ni, wi), torch.where(gp[..., None], nj, wj)
            theta = torch.where(gp, th, theta)
            res = torch.where(act[:, None], torch.stack([r, s], 1), res)
            act = act & ~((r <= tol) & (s <= tol))
            if not bool(act.any()):
                break
            if adapt and (k + 1) % adapt[0] == 0 and k + 1 < iters:
                sc = torch.where(r > adapt[1] * s, adapt[2], torch.where(s > adapt[1] * r, 1.0 / adapt[2], 1.0))
                sc = torch.where(act, sc, torch.ones_like(sc))
                rho = rho * sc
                yi, yj = yi / sc[self.psc][:, None, None], yj / sc[self.psc][:, None, None]
                H, W = self.hessian(rho[self.asc] * self.nc)
        self.u, self.side, self.X, self.theta, self.res = u, side, X, theta, res

    def packed(self):
        x = torch.cat([self.x0[:, None], self.X], 1)
        keep = torch.cat([self.am[:, :1], self.am], 1)
        return dict(X=x[keep].reshape(-1), U=self.u.reshape(self.na, self.Tm, self.nu)[self.am].reshape(-1),
                    theta=self.theta[self.pm], W=None, status=None, iters=None, res=self.res)


def _plain_gradient(b, case, targets):
    """States and gradients at the active set that the plain solve ends with: each scenario's reduced system by
    its dense Schur complement, differentiated by torch."""
    m = _Plain(b, case)
    m.solve(1e-6, int(case["iters"]), adapt=(10, 10.0, 2.0))
    S, n, T, dp = int(case["scen"]), int(case["nmax"]), m.Tm, m.dp
    f = lambda v: torch.tensor(v, dtype=torch.float64, device=m.dev, requires_grad=True)  # noqa: E731
    Q, R, goal = f(b.Qd), f(b.Rd), f(b.x_ref)
    m.q(Q, R, 10.0 * Q, goal)
    H, W = m.hessian(torch.zeros(m.na, dtype=torch.float64, device=m.dev))
    G, free = m.free()
    lin = (G.transpose(1, 2) @ (W * free - m.Q2 * goal[:, None]).reshape(m.na, -1, 1))[..., 0]
    held = m.side != 0
    ub = torch.where(m.side < 0, m.lo, m.hi) * held
    Hm = H * (~held)[:, :, None] * (~held)[:, None, :] + torch.diag_embed(held.to(H.dtype))
    Hi = torch.linalg.inv(Hm) * (~held)[:, :, None] * (~held)[:, None, :]
    rhs = -(lin + (H @ ub[..., None])[..., 0])
    Gp = G.reshape(1, T, m.nx, -1)[0, :, :dp]
    u0 = ub + (Hi @ rhs[..., None])[..., 0]
    us = []
    for s in range(S):
        at = slice(s * n, (s + 1) * n)
        mine = torch.nonzero(m.psc == s)[:, 0]
        pk, tk = torch.nonzero(m.theta[mine] > 1e-9, as_tuple=True)
        if not len(pk):
            us.append(u0[at])
            continue
        pk = mine[pk]
        row = (m.a[pk, tk][:, :, None] * Gp[tk]).sum(1)
        C = torch.zeros(len(pk), n, row.shape[1], dtype=torch.float64, device=m.dev)
        e = torch.arange(len(pk), device=m.dev)
        C[e, m.pi[pk] - s * n] = row
        C[e, m.pj[pk] - s * n] = -row
        off = m.d[s] - (m.a[pk, tk] * (free[m.pi[pk], tk, :dp] - free[m.pj[pk], tk, :dp])).sum(1)
        HC = torch.einsum("iab,mib->mia", Hi[at], C)
        Sc = torch.einsum("mia,kia->mk", C, HC)
        mu = torch.linalg.pinv(0.5 * (Sc + Sc.T), rtol=1e-11, hermitian=True) @ (off - torch.einsum("mia,ia->m", C, u0[at]))
        us.append(u0[at] + torch.einsum("mia,m->ia", HC, mu))
    X = m.states(torch.cat(us))
    pos = X[:, :, :dp].reshape(-1, dp)
    loss = ((pos - torch.tensor(targets, dtype=torch.float64, device=m.dev)) ** 2).sum()
    loss.backward()
    full = torch.cat([m.x0[:, None], X.detach()], 1).reshape(-1)
    # the weights' gradients hang, where rows are all but dependent, on which of them count as such
    return dict(X=full, loss=loss.detach(), gQ=None, gR=None, gGoal=goal.grad)


def exact(case, seed):
    how, it = case.get("run"), int(case["iters"])
    if how in ("polish", "sqp"):
        return None  # which rows are tried next, or linearized where, hangs on the whole path before
    dims = case["tmax"] * (3 if case["kind"] == "swarm" else 2)
    if case["scen"] * case["nmax"] * dims ** 3 / 5e11 * it * 3 + it * 0.02 > 15:
        return None  # more than about 20 seconds
    b = _batch(case, seed)
    if how == "train":
        return _plain_gradient(b, case, b.targets)
    m = _Plain(b, case)
    m.solve(1e-4, it, adapt=(10, 10.0, 2.0) if case.get("adapt") else None, relax=float(case.get("relax", 1.0)))
    return {k: None if v is None else v.cpu() for k, v in m.packed().items()}
