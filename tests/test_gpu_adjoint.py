"""The adjoint's parts at the sizes where their layout changes: one thread per axis
(an agent's axes on the lanes of a warp: 16 agents in 2D, 10 in 3D), the shortest horizons,
more agents than a group holds."""
import numpy as np
import pytest

from instances import random_scenario

pytestmark = pytest.mark.gpu


def _solve(b, flags=0, it=40):
    import paper_2602_15838_gb300 as tg
    s = tg.Solver(b, flags=flags)
    s.solve(0.0, it)
    g = np.random.default_rng(3).standard_normal(s.sizes["X"])
    r = s.backward(g)
    p = s.polish(1e-9, 3)
    q = s.backward(g)
    s.close()
    return r, p, q


@pytest.mark.parametrize("dp,N,T", [(2, 1, 3), (2, 2, 1), (2, 16, 6), (2, 17, 6), (3, 10, 4), (3, 11, 4), (2, 40, 5)])
def test_axis_solves_equal_general_solves(dp, N, T):
    """The double integrator's solves by axis against the general products (the
    same solver with the structure switched off): gradients, polished states and
    the sets after three polishing rounds.  The tolerance is the parity tests' for
    gradients, relative to the largest entry: both form the same sums in float64,
    and the sets here are well conditioned (few rows at these separations)."""
    import paper_2602_15838_gb300 as tg
    b = random_scenario(seed=500 + N + T, N=N, T=T, dp=dp, box=8.0, d_min=0.5)
    (r0, p0, q0), (r1, p1, q1) = _solve(b), _solve(b, tg.FLAG_NO_STRUCTURE)
    for x, y in ((r0, r1), (q0, q1)):
        assert np.array_equal(x["status"], y["status"]) and np.array_equal(x["n_dependent"], y["n_dependent"])
        for k in ("gQ", "gQf", "gR", "gGoal", "X_polished"):
            assert np.abs(x[k] - y[k]).max() <= 1e-6 * max(1.0, np.abs(y[k]).max()), k
    for k in ("act", "W", "status", "rounds"):
        assert np.array_equal(p0[k], p1[k]), k
