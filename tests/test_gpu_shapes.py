"""Agents of a group over the warps of its CTA, and groups packed for few agents."""
import numpy as np
import pytest

from instances import make_batch, make_workload, random_scenario

pytestmark = pytest.mark.gpu


def _run(b, it=10, **kw):
    import paper_2602_15838_gb300 as tg
    s = tg.Solver(b, **kw)
    s.solve(0.0, it)
    out = s.solution()
    cnt = s.counters()
    s.close()
    return out, cnt


@pytest.mark.parametrize("N,dp", [(1, 2), (16, 2), (17, 2), (31, 2), (32, 2), (10, 3), (11, 3), (21, 3), (32, 3)])
def test_agents_over_warps(N, dp):
    """Every number of warps gives the same bits and counts: the agent counts at
    which another warp is taken (16 per warp in 2D, 10 in 3D) and the most."""
    b = random_scenario(seed=40 + N, N=N, T=6, dp=dp, box=6.0, umax=0.7)
    ref, cref = _run(b, threads_per_cta=32)
    for t in (64, 96, 128, 256):
        g, c = _run(b, threads_per_cta=t)
        for k in ("X", "U", "theta", "W", "status", "iters", "res"):
            assert np.array_equal(g[k], ref[k]), (t, k)
        assert np.array_equal(c["eqp"], cref["eqp"]) and np.array_equal(c["fact"], cref["fact"]), t


@pytest.mark.parametrize("n_scen,adapt,relax", [(3, None, 1.0), (40, (5, 10.0, 2.0), 1.0), (40, None, 1.5), (300, None, 1.0)])
def test_packing_by_batch_size(n_scen, adapt, relax):
    """Scenarios give the same bits in a batch of any size, that is in groups of
    any size: alone, in a small batch and in a larger one."""
    b = make_workload("mixed", n_scen=n_scen, first=50)
    big = make_workload("mixed", n_scen=1400, first=50) if n_scen == 300 else None
    g, _ = _run(b, adapt=adapt, relax=relax)
    xo = np.concatenate([[0], np.cumsum(b.N.astype(int) * (b.T + 1) * b.nx)])
    to = np.concatenate([[0], np.cumsum(b.P * b.T)])
    for k in range(0, n_scen, max(1, n_scen // 5)):
        o, _ = _run(b.scenario(k), adapt=adapt, relax=relax)
        assert np.array_equal(o["X"], g["X"][xo[k]:xo[k + 1]]) and np.array_equal(o["theta"], g["theta"][to[k]:to[k + 1]]), k
    if big is not None:
        h, _ = _run(big)
        assert np.array_equal(h["X"][:xo[-1]], g["X"]) and np.array_equal(h["theta"][:to[-1]], g["theta"])
