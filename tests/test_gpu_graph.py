"""The graph mode's kernels after the x-update (partner masks, one CTA per small
scenario) against the persistent kernel, which they equal bit for bit."""
import numpy as np
import pytest

from instances import make_batch, nearest_neighbour_pairs, random_scenario

pytestmark = pytest.mark.gpu


def _batch(sizes, d, dp=2):
    parts = []
    for k, (N, T) in enumerate(sizes):
        s = random_scenario(seed=70 + 3 * k + N, N=N, T=T, dp=dp, box=8.0)
        parts.append(dict(N=N, T=T, x_init=s.x_init, x_ref=s.x_ref, a=s.a, w0=s.w0, d=d, rho=1.0, umax=1.0, c=None))
    return make_batch(parts, dp=dp, dt=0.1, umax=1.0)


def _run(b, tol, it, **kw):
    import paper_2602_15838_gb300 as tg
    s = tg.Solver(b, **kw)
    outs = []
    for _ in range(2):      # the second solve finds what the first left in its buffers
        s.solve(tol, it)
        outs.append(s.solution())
    s.close()
    assert all(np.array_equal(outs[0][k], outs[1][k]) for k in ("X", "U", "theta", "W", "status", "iters", "res"))
    return outs[0]


# one small scenario, small ones of several horizons (one CTA each), a word of partners and just
# more, and a batch that mixes them (grid-wide kernels); none, some and all halfspaces pushing
@pytest.mark.parametrize("sizes", [((2, 3),), ((32, 4), (1, 2), (13, 7)), ((33, 3),), ((64, 3),), ((70, 4), (5, 2))])
@pytest.mark.parametrize("d", [-50.0, 0.4, 20.0])
@pytest.mark.parametrize("precision", [64, 32])
def test_graph_equals_batched(sizes, d, precision):
    b = _batch(sizes, d)
    for tol, it in ((0.0, 7), (1e-2, 60)):
        ref = _run(b, tol, it, precision=precision)
        g = _run(b, tol, it, precision=precision, mode="graph")
        for k in ("X", "U", "theta", "W", "status", "iters"):
            assert np.array_equal(g[k], ref[k]), (tol, k)
        assert np.abs(g["res"] - ref["res"]).max() <= (1e-12 if precision == 64 else 1e-5) * max(1.0, ref["res"].max())


def test_graph_listed_pairs_and_3d():
    for b in (nearest_neighbour_pairs(_batch(((20, 5), (9, 4)), 1.0), 3), nearest_neighbour_pairs(_batch(((40, 3),), 1.0), 3),
              _batch(((12, 4), (34, 3)), 0.8, dp=3)):
        ref, g = _run(b, 0.0, 8), _run(b, 0.0, 8, mode="graph")
        for k in ("X", "U", "theta", "W"):
            assert np.array_equal(g[k], ref[k]), k
