"""One ragged row of large tiles (31 of its 32 rows exist), bit for bit against
the oracle: a launch takes them from 3 x 152 tiles on, so one row needs more
than 14,560 columns in some bit's set."""
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_grid import dev, same

pytestmark = pytest.mark.gpu


def set_count(T, bit):
    """Exponents 1..T with this bit: the columns of its product."""
    return sum((e >> bit) & 1 for e in range(1, T + 1))


@pytest.mark.parametrize("qf", [4.0, -1.0])
@pytest.mark.parametrize("T", [29185, 30001])  # 14592 + columns: 456 tiles and a few more
def test_one_row_of_large_tiles(T, qf):
    import paper_2212_11744_gb300 as lqt
    G = 31
    assert max(-(-set_count(T, b) // 32) for b in range(T.bit_length())) >= 3 * 152
    g = W.falling_body(G=G, T=T)
    g.qf = qf
    Vb = oracle.grid_block(g)
    got = lqt.lqt_grid_values(g, dev(Vb))
    torch.cuda.synchronize()
    assert lqt.lqt_get_status() == 0
    same(got, oracle.grid_values(g, Vb), "values")
