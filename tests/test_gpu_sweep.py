"""The group sweep of the persistent kernel (pairs that do not push are left out)
against the plain sweeps over all pairs, which it must equal bit for bit."""
import dataclasses

import numpy as np
import pytest

from instances import make_batch, nearest_neighbour_pairs, random_scenario

pytestmark = pytest.mark.gpu


def _run(b, it=12, **kw):
    import paper_2602_15838_gb300 as tg
    s = tg.Solver(b, **kw)
    s.solve(0.0, it)
    out = s.solution()
    s.close()
    return out


def _batch(sizes, T, dp=2, d=0.4, scale=1.0):
    parts = []
    for k, N in enumerate(sizes):
        s = random_scenario(seed=300 + 7 * k + N, N=N, T=T, dp=dp, box=6.0)
        parts.append(dict(N=N, T=T, x_init=scale * s.x_init, x_ref=scale * s.x_ref, a=s.a, w0=scale * s.w0, d=d, rho=1.0,
                          umax=1.0, c=None))
    return make_batch(parts, dp=dp, dt=0.1, umax=1.0)


# pairs of a group around the batch of 4 x 32 (16 agents: 120, 17: 136) up to 32 agents (496),
# several members, a lone agent; separations where no, some and all halfspaces push
@pytest.mark.parametrize("sizes,dp", [((2,), 2), ((16,), 2), ((17,), 2), ((32,), 2), ((1, 3, 12, 16), 2), ((9, 8, 8, 7), 3)])
@pytest.mark.parametrize("d", [-50.0, 0.4, 30.0])
@pytest.mark.parametrize("precision", [64, 32])
def test_sweep_equals_plain_sweeps(sizes, dp, d, precision):
    import paper_2602_15838_gb300 as tg
    b = _batch(sizes, 5, dp=dp, d=d)
    ref = _run(b, precision=precision, flags=tg.FLAG_NO_FUSED_PAIR_GATHER)
    for kw in (dict(threads_per_cta=32), dict(threads_per_cta=128)):
        g = _run(b, precision=precision, **kw)
        for k in ("X", "U", "theta", "W", "status", "iters"):
            assert np.array_equal(g[k], ref[k]), (kw, k)


def test_sweep_with_listed_pairs_and_far_positions():
    """Listed pairs (an agent's partners by its list) and positions at which the
    float32 test has no say (beyond 2^60) or sits within its own error."""
    import paper_2602_15838_gb300 as tg
    b = nearest_neighbour_pairs(_batch((12, 7, 13), 6, d=1.2), 3)
    far = _batch((6, 5), 6, scale=1e19)
    near = _batch((14,), 6)
    # separations equal to the first step's own distances: g at its rounding
    diff = near.w0.reshape(14, 6, 2)[0, 0] - near.w0.reshape(14, 6, 2)[1, 0]
    near = dataclasses.replace(near, d_min=np.array([float(np.sqrt((diff ** 2).sum()))]))
    for c in (b, far, near):
        ref = _run(c, flags=tg.FLAG_NO_FUSED_PAIR_GATHER)
        g = _run(c)
        for k in ("X", "U", "theta", "W", "status", "iters"):
            assert np.array_equal(g[k], ref[k]), k
