"""The n = 64 element build by repeated sub-interval lengths (the mixed-precision
solve of constant F, L, U, X) against the mixed solve of the same problem whose
F is given per sub-interval, which builds element by element: the same bits.
Lengths: one; the rounding of an equal grid; three interleaved; more lengths than
kept products (152); all different; and T at the edges of the search's CTAs."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.test_gpu_uniform import make, with_grid

pytestmark = pytest.mark.gpu


def grid(kind, T, rng):
    if kind == "one":
        return np.arange(T + 1) / 32.0
    if kind == "equal":
        return np.linspace(0.3, 0.3 + 0.04 * T, T + 1)
    if kind == "three":
        return np.concatenate([[0.0], np.cumsum(np.array([1.0, 1.5, 1.25])[np.arange(T) % 3] / 32.0)])
    if kind == "many":  # 200 lengths, each once or more
        return np.concatenate([[0.0], np.cumsum((512 + rng.permutation(np.arange(T) % 200)) / 16384.0)])
    return np.concatenate([[0.0], np.cumsum(rng.uniform(0.02, 0.06, T))])


@pytest.mark.parametrize("kind,T,K,r", [("one", 128, 1, "interval"), ("equal", 129, 2, "const"),
                                        ("three", 257, 3, "interval"), ("many", 300, 1, "interval"),
                                        ("many", 300, 8, "none"), ("all", 160, 2, "const")])
def test_mixed_solve_same_bits(kind, T, K, r):
    import paper_2212_11744_gb300 as lqt
    rng = np.random.default_rng(T + K)
    p = make(64, 16, T, K, "equal", r)
    p.F = W.const(p.F.values.reshape(64, 64) * 0.5)
    p.t = grid(kind, T, rng)
    a = lqt.lqt_solve_mixed(lqt.DeviceProblem(p))
    torch.cuda.synchronize()
    assert lqt.lqt_get_status() == 0
    p.F = W.Coef(np.repeat(p.F.values.reshape(1, 64, 64), T, 0), W.PER_INTERVAL)
    b = lqt.lqt_solve_mixed(lqt.DeviceProblem(p))
    torch.cuda.synchronize()
    assert lqt.lqt_get_status() == 0
    for k in a:
        assert torch.equal(a[k], b[k]), k
