"""Graph mode on either side of the line between one tail CTA per scenario and grid-wide
kernels ((pairs + agents) x steps of the largest scenario against 2560), at short and long
horizons: the iterates of the batched mode, bit for bit."""
import numpy as np
import pytest

from instances import make_batch, nearest_neighbour_pairs, random_scenario

pytestmark = pytest.mark.gpu


def _batch(sizes, dp=2):
    parts = []
    for k, (N, T) in enumerate(sizes):
        s = random_scenario(seed=700 + 11 * k + N, N=N, T=T, dp=dp, box=6.0)
        parts.append(dict(N=N, T=T, x_init=s.x_init, x_ref=s.x_ref, a=s.a, w0=s.w0, d=0.8, rho=1.0, umax=1.0, c=None))
    return make_batch(parts, dp=dp, dt=0.1, umax=1.0)


@pytest.mark.parametrize("sizes,dp,knn", [(((14, 24),), 2, 0), (((14, 25),), 2, 0), (((32, 4),), 2, 0), (((32, 5), (3, 9)), 2, 0),
                                          (((3, 300),), 2, 0), (((3, 500),), 2, 0), (((12, 40),), 3, 0), (((32, 60),), 2, 3),
                                          (((2, 860), (1, 3)), 2, 0)])
@pytest.mark.parametrize("precision", [64, 32])
def test_graph_tail_and_grid_equal_batched(sizes, dp, knn, precision):
    import paper_2602_15838_gb300 as tg
    b = _batch(sizes, dp)
    if knn:
        b = nearest_neighbour_pairs(b, knn)
    out = []
    for mode in ("batched", "graph"):
        s = tg.Solver(b, precision=precision, mode=mode)
        for _ in range(2):      # the second solve finds what the first left in its buffers
            s.solve(0.0, 6)
            out.append(s.solution())
        s.close()
    for g in out[1:]:
        for k in ("X", "U", "theta", "W", "status", "iters"):
            assert np.array_equal(g[k], out[0][k]), k
