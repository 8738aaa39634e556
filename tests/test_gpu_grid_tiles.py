"""The two tile sizes of the grid products at their edges, bit for bit against
the oracle: grids around one tile row, around the largest staged reduction
(224 points) and beyond it; the bounds of nonnegative operands, of operands of
both signs, and of operands outside the screen's range."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_grid import dev, same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,T", [
    (31, 20001), (33, 19999), (65, 14001),  # 1, 2, 3 rows of large tiles, ragged columns
    (224, 5600), (225, 4900), (300, 4000),  # one stage, one stage and 1, one stage and 76
])
@pytest.mark.parametrize("qf", [4.0, -1.0])
def test_values_in_large_tiles(G, T, qf):
    import paper_2212_11744_gb300 as lqt
    g = W.falling_body(G=G, T=T)
    g.qf = qf  # a negative terminal cost: operands of both signs
    Vb = oracle.grid_block(g)
    got = lqt.lqt_grid_values(g, dev(Vb))
    torch.cuda.synchronize()
    assert lqt.lqt_get_status() == 0
    same(got, oracle.grid_values(g, Vb), "values")


@pytest.mark.parametrize("G", [15, 17, 223, 226, 449, 1100])  # 1100: 35 x 35 large tiles
@pytest.mark.parametrize("kind", ["positive", "signs", "range", "zeros"])
def test_combine_at_tile_edges(G, kind):
    import paper_2212_11744_gb300 as lqt
    g = W.falling_body(G=G, T=1)
    rng = np.random.default_rng(G)
    x = g.grid()
    A = (x[:, None] - 0.4 * x[None, :]) ** 2 + rng.uniform(0.0, 0.3, (G, G))
    B = 0.8 * (x[:, None] - x[None, :]) ** 2 + rng.uniform(0.0, 0.3, (G, G))
    if kind == "signs":
        B[-1, -1] = -0.25  # the last tile alone
    elif kind == "range":
        A[G - 1, G // 2] = 2e30  # above 2^100: the last row of tiles
    elif kind == "zeros":
        A[:, ::3], B[::3] = 0.0, -0.0
    got = lqt.lqt_grid_combine(g, dev(A), dev(B))
    torch.cuda.synchronize()
    assert lqt.lqt_get_status() == 0
    same(got, oracle.grid_combine(g, A, B), kind)
