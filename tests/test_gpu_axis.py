"""The double integrator's per-axis recursions at the agent counts where the lane
layout changes (one lane per axis holds 16 agents of a warp in 2D, 10 in 3D) and at
the shortest horizons."""
import numpy as np
import pytest

from instances import heterogeneous_agents, make_batch, random_scenario

pytestmark = pytest.mark.gpu


def _one(dp, N, T, seed):
    return random_scenario(seed=seed, N=N, T=T, dp=dp, box=6.0, umax=0.6)


def _run(b, **kw):
    import paper_2602_15838_gb300 as tg
    s = tg.Solver(b, **kw)
    s.solve(0.0, 9)
    out = s.solution()
    cnt = s.counters()
    s.close()
    return out, cnt


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("dp,N,T", [(2, 1, 1), (2, 2, 2), (2, 16, 7), (2, 17, 7), (2, 32, 12), (3, 1, 1), (3, 10, 7),
                                    (3, 11, 7), (3, 32, 9)])
def test_axis_recursions(dp, N, T, precision):
    """One lane per axis and one lane per agent give the same bits and counts, in
    the batched and the graph mode; the general dense products give the same
    working sets and, in float64, the same iterates to 1e-12 (nine iterations of
    rounding of a few ulp of well conditioned stages)."""
    import paper_2602_15838_gb300 as tg
    b = _one(dp, N, T, seed=100 * dp + N)
    ref, cref = _run(b, precision=precision, flags=tg.FLAG_NO_LANE_GROUPS)
    for kw in (dict(), dict(threads_per_cta=32), dict(mode="graph"), dict(mode="graph", flags=tg.FLAG_NO_LANE_GROUPS)):
        g, c = _run(b, precision=precision, **kw)
        for k in ("X", "U", "theta", "W", "status", "iters"):
            assert np.array_equal(g[k], ref[k]), (kw, k)
        assert np.array_equal(c["eqp"], cref["eqp"]) and np.array_equal(c["fact"], cref["fact"]), kw
    if precision == 64:
        d, cd = _run(b, flags=tg.FLAG_NO_STRUCTURE)
        assert np.array_equal(d["W"], ref["W"]) and np.array_equal(cd["eqp"], cref["eqp"])
        for k in ("X", "U", "theta"):
            assert np.abs(d[k] - ref[k]).max(initial=0.0) <= 1e-12 * max(1.0, np.abs(ref[k]).max(initial=0.0)), k


def test_large_magnitudes_and_held_multipliers():
    """Weights and goals far from one: the float32 sign test of the multipliers
    must hand over to float64 where its numbers leave float32's range, and the
    result is the one of the dense products."""
    import paper_2602_15838_gb300 as tg
    b = _one(2, 6, 10, seed=5)
    for f in (1e-30, 1e25):
        c = make_batch([dict(N=6, T=10, x_init=b.x_init, x_ref=b.x_ref, a=b.a, w0=b.w0, d=0.4, rho=f, umax=0.6, c=None)],
                       dp=2, dt=0.1, umax=0.6, q_pos=f, q_vel=0.1 * f, r=0.1 * f)
        g, cg = _run(c)
        d, cd = _run(c, flags=tg.FLAG_NO_STRUCTURE)
        assert np.array_equal(g["W"], d["W"]) and np.array_equal(cg["eqp"], cd["eqp"])
        assert np.abs(g["X"] - d["X"]).max() <= 1e-12 * np.abs(d["X"]).max()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("dp,N,T", [(2, 1, 3), (2, 16, 7), (2, 17, 7), (3, 11, 6)])
def test_axis_recursions_per_agent_models(dp, N, T, precision):
    """Agents of unlike mass and damping: the per-axis recursions give the bits of the
    dense products, in both modes; and after an update to models that couple the
    axes (and back) the handle takes the products that these need."""
    import dataclasses

    import paper_2602_15838_gb300 as tg
    b = heterogeneous_agents(_one(dp, N, T, seed=31 + N), seed=4)
    ref, cref = _run(b, precision=precision, flags=tg.FLAG_NO_STRUCTURE)
    for kw in (dict(), dict(flags=tg.FLAG_NO_LANE_GROUPS), dict(mode="graph")):
        g, c = _run(b, precision=precision, **kw)
        for k in ("X", "U", "theta", "W", "status", "iters"):
            assert np.array_equal(g[k], ref[k]), (kw, k)
        assert np.array_equal(c["eqp"], cref["eqp"]), kw
    A2 = b.A_agent.copy()
    A2[:, 0, 1] = 0.01
    mixed = dataclasses.replace(b, A_agent=A2)
    want, _ = _run(mixed, precision=precision, flags=tg.FLAG_NO_STRUCTURE)
    s = tg.Solver(b, precision=precision)
    for data, exp in ((b, ref), (mixed, want), (b, ref)):
        s.update(data)
        s.solve(0.0, 9)
        out = s.solution()
        assert np.array_equal(out["X"], exp["X"]) and np.array_equal(out["W"], exp["W"])
    s.close()


@pytest.mark.parametrize("dp,N,T", [(2, 3, 16), (2, 5, 33), (3, 4, 22), (2, 2, 70), (3, 18, 5)])
@pytest.mark.parametrize("start", ["turbo", "cold"])
def test_ratio_test_over_the_lanes(dp, N, T, start):
    """The ratio test that spreads an agent's inputs over the lanes (32 and 64 of
    them are the edges of what it keeps in registers) blocks on the same inputs as
    the general code's test in index order: the same counts and working sets on
    tight boxes, where most rounds block."""
    import paper_2602_15838_gb300 as tg
    b = random_scenario(seed=11 * N + T, N=N, T=T, dp=dp, box=6.0, umax=0.15)
    g, cg = _run(b, start=start)
    d, cd = _run(b, start=start, flags=tg.FLAG_NO_STRUCTURE)
    assert np.array_equal(cg["eqp"], cd["eqp"]) and np.array_equal(g["W"], d["W"])
    for k in ("X", "U", "theta"):
        assert np.abs(d[k] - g[k]).max(initial=0.0) <= 1e-11 * max(1.0, np.abs(d[k]).max(initial=0.0)), k
    h, ch = _run(b, start=start, mode="graph")
    assert np.array_equal(h["X"], g["X"]) and np.array_equal(ch["eqp"], cg["eqp"])


@pytest.mark.parametrize("dp,N,T", [(2, 2, 63), (2, 2, 64), (2, 2, 65), (3, 2, 42), (3, 2, 43)])
@pytest.mark.parametrize("start", ["turbo", "cold"])
def test_ratio_test_at_the_edge_of_its_registers(dp, N, T, start):
    """The ratio test over the lanes keeps 128 inputs of an agent in registers (four per
    lane) and loads them again beyond: 126 to 130 of them, as above."""
    test_ratio_test_over_the_lanes(dp, N, T, start)
