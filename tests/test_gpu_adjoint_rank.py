"""The adjoint's dense algebra (Schur complement, pivoted factor, least squares) against
the oracle's dense KKT gradient, on active sets whose number of rows and rank are known:
on either side of a warp's lanes (31, 32, 33), of a tile of the normal matrix, beyond the
256 threads of a CTA, and with many more rows than their rank."""
import dataclasses

import numpy as np
import pytest

import oracle
from instances import make_batch, pair_list, random_scenario

pytestmark = pytest.mark.gpu


def _batch(N, T, dp, umax, pairs=None):
    """One scenario whose halfspaces (separation 30) all push in the first iteration."""
    s = random_scenario(seed=1, N=N, T=T, dp=dp, box=6.0)
    b = make_batch([dict(N=N, T=T, x_init=s.x_init, x_ref=s.x_ref, a=s.a, w0=s.w0, d=30.0, rho=1.0, umax=umax, c=None)],
                   dp=dp, dt=0.1, umax=umax)
    if pairs is None:
        return b
    at = {tuple(p): k for k, p in enumerate(pair_list(N))}
    rows = b.a.reshape(len(at), T, dp)[[at[p] for p in pairs]]
    return dataclasses.replace(b, a=np.ascontiguousarray(rows.reshape(-1, dp)), pair_count=np.array([len(pairs)], np.int32),
                               pair_ij=np.array(pairs, np.int32))


def _clusters(fours, twos):
    """Pairs of `fours` groups of four agents, all coupled (6 rows of rank 5 a step in
    2D), and of `twos` couples."""
    p = [(4 * c + i, 4 * c + j) for c in range(fours) for i in range(4) for j in range(i + 1, 4)]
    p += [(4 * fours + 2 * e, 4 * fours + 2 * e + 1) for e in range(twos)]
    return 4 * fours + 2 * twos, p


def _case(kind, n, T, dp):
    # boxes wide enough that no input is held: one step has to undo the whole starting velocity
    umax = 1e4 if T == 1 else 50.0
    if kind == "all":
        return _batch(n, T, dp, umax)
    N, pairs = _clusters(*n)
    return _batch(N, T, dp, umax, pairs)


def _rel(a, b):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / max(1.0, np.abs(np.asarray(b)).max()))


# Tolerance in float64, for states and gradients: the rounding of a block of k coupled rows, k eps over
# the smallest kept eigenvalue of S relative to the largest.  The worst are the couples over many steps
# (33 rows at 4.7e-8: 1.6e-7), below 1e-6 as all others.  In float32 (one step; 37 rows at 5e-3: 4e-4) the
# gradients' usual 1e-3.
@pytest.mark.parametrize("kind,n,T,dp,m,dep,precision", [
    ("all", 2, 31, 2, 31, 0, 64), ("all", 2, 32, 2, 32, 0, 64), ("all", 2, 33, 2, 33, 0, 64),     # full rank
    ("twos", (0, 10), 13, 2, 130, 0, 64), ("twos", (0, 10), 30, 2, 300, 0, 64),
    ("fours", (6, 1), 1, 2, 37, 6, 64), ("fours", (6, 2), 1, 2, 38, 6, 64), ("fours", (6, 3), 1, 2, 39, 6, 64),
    ("fours", (2, 1), 3, 2, 39, 6, 64),
    ("all", 8, 5, 2, 140, 75, 64), ("all", 12, 5, 2, 330, 225, 64), ("all", 24, 1, 2, 276, 231, 64),
    ("all", 9, 5, 3, 180, 75, 64), ("all", 9, 8, 3, 288, 120, 64),
    ("fours", (6, 1), 1, 2, 37, 6, 32), ("fours", (6, 2), 1, 2, 38, 6, 32), ("fours", (6, 3), 1, 2, 39, 6, 32),
    ("all", 24, 1, 2, 276, 231, 32), ("all", 24, 1, 3, 276, 210, 32)])
def test_gradient_at_known_rank(kind, n, T, dp, m, dep, precision):
    import paper_2602_15838_gb300 as tg
    b = _case(kind, n, T, dp)
    N = int(b.N[0])
    s = tg.Solver(b, precision=precision)
    s.solve(0.0, 1)
    out = s.split(s.solution())[0]
    act = out["theta"] > 1e-9
    assert int(act.sum()) == m and not out["W"].any()
    targets = np.random.default_rng(7).uniform(-5.0, 5.0, (N, T, dp))
    X = s.backward(None)["X_polished"].reshape(N, T + 1, 2 * dp)
    gX = np.zeros_like(X)
    gX[:, 1:, :dp] = 2.0 * (X[:, 1:, :dp] - targets)
    g = s.backward(gX.ravel())
    s.close()
    ref = oracle.global_gradient(b, 0, act.astype(np.uint8), out["W"], targets, qf_tie=10.0)
    assert ref["n_dependent"] == dep and int(g["n_dependent"][0]) == dep and int(g["status"][0]) == 0
    tol = 1e-6 if precision == 64 else 1e-3
    assert _rel(X, ref["X"]) <= tol
    assert _rel(g["gQ"] + 10.0 * g["gQf"], ref["gQ"]) <= tol
    assert _rel(g["gR"], ref["gR"]) <= tol
    assert _rel(g["gGoal"], ref["gGoal"]) <= tol
