"""The constant-coefficient build on grids whose steps lie around their mean within
and beyond the table's 1e-9 (offsets in opposite pairs, so that the mean is the
middle one and the table is used): elements, batches and gradients.  An element's
own change over 9e-10 of its step is above the 1e-11 bound, so the table's
first-order term is held to a hundredth of itself."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import TOL, relerr as rel, to_np
from tests.test_gpu_uniform import lqt, make, with_grid

pytestmark = pytest.mark.gpu


def paired_steps(T, h, rng):
    o = rng.choice([0.0, 1e-13, 3e-11, 9e-10, 9e-10, 1.2e-9, 1e-8], T // 2)
    d = np.concatenate([o, -o, np.zeros(T % 2)])
    return h * (1.0 + rng.permutation(d))


def served(t, K):
    """Sub-intervals within 1e-9 of the mean step."""
    h0 = (t[-1] - t[0]) / ((len(t) - 1) * K)
    return np.abs(np.diff(t) / K - h0) <= 1e-9 * h0


def problem(n, m, T, K, seed=0):
    p = make(n, m, T, K, "equal", "interval")
    with_grid(p, paired_steps(T, 0.04, np.random.default_rng(seed + n + T)))
    near = served(p.t, K)
    assert near.mean() > 0.55 and not near.all()
    return p


@pytest.mark.parametrize("n,m,T,K", [(1, 1, 32769, 3), (2, 1, 32800, 4), (3, 2, 32770, 2), (4, 2, 8193, 4),
                                     (8, 4, 1100, 4), (16, 8, 530, 4), (64, 16, 131, 2)])
def test_elements(n, m, T, K):
    p = problem(n, m, T, K)
    el = lqt().lqt_build_elements(lqt().DeviceProblem(p))
    torch.cuda.synchronize()
    assert lqt().lqt_get_status() == 0
    for j0, j1 in ((0, min(T + 1, 96)), (max(0, T - 40), T + 1)):
        ref = oracle.build_elements(p, j0, j1)
        for k in ("A", "b", "C", "eta", "J", "zeta"):
            assert rel(to_np(el[k][j0:j1]), ref[k]) <= 1e-11, (k, j0)


@pytest.mark.parametrize("n", [3, 8, 16])
def test_batch(n):
    from paper_2212_11744_gb300.batch import Batch
    ps = [problem(n, max(1, n // 2), T, 4, seed=T) for T in (64, 65, 200, 1000)]
    b = Batch(ps)
    out = b.solve()
    torch.cuda.synchronize()
    for i, p in enumerate(ps):
        ref, got = oracle.solve(p), b.problem_slice(out, i)
        for k in ("S", "v", "zeta", "x", "u"):
            assert rel(to_np(got[k]), ref[k]) <= TOL, (i, k)


@pytest.mark.parametrize("K", [1, 4])
def test_gradients(K):
    from tests.test_gpu_adjoint import TOL as GTOL, gpu_grads, oracle_grads, rel as grel, weights
    p = problem(8, 4, 1056, K)
    w = weights(p, 5)
    got, ref = gpu_grads(p, *w), oracle_grads(p, *w)
    for k in ref:
        assert grel(got[k].reshape(ref[k].shape), ref[k]) <= GTOL, k


@pytest.mark.parametrize("n", [2, 4])
def test_gradients_beyond_one_segment(n):
    """Constant F (the shared element) against the same F per sub-interval."""
    from tests.test_gpu_adjoint import TOL as GTOL, gpu_grads, rel as grel
    T = 33001
    p = problem(n, 1, T, 2)
    rng = np.random.default_rng(n)
    w = (rng.standard_normal((T + 1, n, n)), rng.standard_normal((T + 1, n)), rng.standard_normal(T + 1),
         rng.standard_normal((T + 1, n)), 1.3)
    a = gpu_grads(p, *w)
    p.F = W.Coef(np.repeat(p.F.values, T, axis=0), W.PER_INTERVAL)
    b = gpu_grads(p, *w)
    b["F"] = b["F"].sum(axis=0, keepdims=True)
    for k in a:
        assert grel(a[k], b[k]) <= GTOL, k
