"""Constant coefficients on a (nearly) uniform grid: the element build from one
integrated element (csrc/lqt_uniform.cu) against the oracle's RK4 of every
sub-interval.  Bound 1e-11 per element, as for the general build: both sides
take the same RK4 steps, the table drops terms below (1e-9)^2 relative, and
the rest is FP64 rounding of sums of at most a few hundred terms."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import TOL, relerr as rel, to_np

pytestmark = pytest.mark.gpu


def lqt():
    import paper_2212_11744_gb300 as m
    return m


def with_grid(p, steps):
    p.t = np.concatenate([[0.3], 0.3 + np.cumsum(steps)])
    return p


def steps_of(kind, T, h, rng):
    """Sub-interval lengths: equal; equal up to small relative offsets on both
    sides of the 1e-9 line; every third one another length; all different."""
    d = np.full(T, h)
    if kind == "offsets":
        d *= 1.0 + rng.choice([0.0, 1e-13, -3e-11, 9e-10, -9e-10, 1.1e-9, -1e-8], T)
    elif kind == "thirds":
        d[::3] *= rng.uniform(0.5, 1.5)
    elif kind == "uneven":
        d *= rng.uniform(0.5, 1.5, T)
    return d


CASES = [  # n, m, T, K, grid, r
    (1, 1, 32768, 3, "equal", "interval"), (2, 1, 32801, 4, "offsets", "interval"), (3, 2, 32769, 2, "thirds", "const"),
    (4, 2, 8192, 4, "equal", "interval"), (4, 4, 8255, 1, "uneven", "interval"), (4, 1, 8191, 4, "offsets", "interval"),
    (8, 4, 1024, 4, "offsets", "interval"), (8, 8, 1087, 2, "thirds", "none"), (8, 3, 1025, 3, "equal", "const"),
    (16, 8, 512, 4, "offsets", "interval"), (16, 16, 527, 1, "thirds", "const"), (16, 1, 513, 2, "equal", "none"),
    (64, 16, 128, 2, "offsets", "interval"), (64, 5, 143, 1, "thirds", "none"),
]


def make(n, m, T, K, grid, r, H=False):
    rng = np.random.default_rng(1000 * n + m + T)
    p = W.batched_member(11 + n, T=T, n=n)
    G = rng.standard_normal((m, m))
    p.m, p.K = m, K
    p.L = W.const(rng.standard_normal((n, m)) / np.sqrt(n))
    p.U = W.const(G @ G.T + 0.3 * np.eye(m))
    if r == "const":
        p.r = W.const(rng.standard_normal(n))
    elif r == "none":
        p.r = None
    if H:
        nr = max(1, n - 1)
        X = rng.standard_normal((nr, nr))
        p.nr, p.H, p.Hf = nr, W.const(rng.standard_normal((nr, n))), rng.standard_normal((nr, n))
        p.X, p.Xf, p.rf = W.const(X @ X.T + 0.1 * np.eye(nr)), np.eye(nr), rng.standard_normal(nr)
        p.r = W.Coef(rng.standard_normal((T, nr)), W.PER_INTERVAL)
    return with_grid(p, steps_of(grid, T, 0.04, rng))


@pytest.mark.parametrize("n,m,T,K,grid,r", CASES)
def test_elements_match_oracle(n, m, T, K, grid, r):
    p = make(n, m, T, K, grid, r)
    el = lqt().lqt_build_elements(lqt().DeviceProblem(p))
    torch.cuda.synchronize()
    assert lqt().lqt_get_status() == 0
    spans = [(0, min(T + 1, 96)), (max(0, T - 40), T + 1)]
    for j0, j1 in spans:
        ref = oracle.build_elements(p, j0, j1)
        for k in ("A", "b", "C", "eta", "J", "zeta"):
            assert rel(to_np(el[k][j0:j1]), ref[k]) <= 1e-11, (k, j0)


@pytest.mark.parametrize("n", [4, 16])
def test_output_matrix_and_mixed_path(n):
    """With H; the mixed-precision solve keeps the general build (its elements
    agree with the FP64 solve to its own 1e-4 target)."""
    p = make(n, 2, {4: 8200, 16: 530}[n], 2, "offsets", "interval", H=True)
    dp = lqt().DeviceProblem(p)
    out, mix = lqt().lqt_solve(dp), lqt().lqt_solve_mixed(dp)
    ref = oracle.solve(p)
    for k in ("S", "v", "zeta", "x", "u"):
        assert rel(to_np(out[k]), ref[k]) <= TOL, k
        a, b = to_np(mix[k]), ref[k]
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max(), k


def test_host_call_equals_device_call():
    p = make(4, 2, (1 << 16) + 5, 4, "offsets", "interval")
    m = lqt()
    dev = m.lqt_solve(m.DeviceProblem(p))
    hp = m.HostProblem(p)
    ws = torch.empty(m.lqt_workspace_size(hp, m.LQT_WS_SOLVE) + m.lqt_host_staging_size(hp) + 4096,
                     dtype=torch.uint8, device="cuda")
    host = m.lqt_solve_host(hp, ws)
    for k in ("S", "v", "zeta", "x", "u", "cost"):
        np.testing.assert_array_equal(host[k].numpy(), to_np(dev[k]))


@pytest.mark.parametrize("n", [2, 4, 8, 16])
def test_batch_members_with_other_grids(n):
    """Members short and long, uniform and not, one with a drift (which keeps
    the general build)."""
    from paper_2212_11744_gb300.batch import Batch
    rng = np.random.default_rng(n)
    Ts = [1, 63, 64, 65, 200, 129]
    probs = [W.batched_member(50 * n + i, T=T, n=n) for i, T in enumerate(Ts)]
    for p, kind in zip(probs, ("equal", "equal", "offsets", "thirds", "uneven", "equal")):
        with_grid(p, steps_of(kind, p.T, 0.05, rng))
    probs[5].c = W.const(rng.standard_normal(n))
    bt = Batch(probs)
    out = bt.solve()
    torch.cuda.synchronize()
    for b, p in enumerate(probs):
        ref, got = oracle.solve(p), bt.problem_slice(out, b)
        for k in ("S", "v", "zeta", "x", "u"):
            assert rel(to_np(got[k]), ref[k]) <= TOL, (b, k)


@pytest.mark.parametrize("grid,r,K", [("equal", "interval", 4), ("offsets", "interval", 2), ("thirds", "interval", 1),
                                      ("offsets", "const", 8), ("uneven", "interval", 2)])
def test_gradients_match_oracle(grid, r, K):
    """The reverse sweep of the shared element (csrc/lqt_uniform_adjoint.cu)
    beside the sweeps of the sub-intervals it does not serve."""
    from tests.test_gpu_adjoint import TOL as GTOL, gpu_grads, oracle_grads, rel as grel, weights
    p = make(8, 4, 1027 if K == 4 else 1056, K, grid, r)
    w = weights(p, 5)
    got, ref = gpu_grads(p, *w), oracle_grads(p, *w)
    for k in ref:
        assert grel(got[k].reshape(ref[k].shape), ref[k]) <= GTOL, k


@pytest.mark.parametrize("n", [2, 4])
def test_gradients_beyond_one_segment(n):
    """T above the reverse sweep's segment: constant F (the shared element)
    against the same F given per sub-interval (the general sweeps)."""
    from tests.test_gpu_adjoint import TOL as GTOL, gpu_grads, rel as grel
    T = 33001
    p = make(n, 1, T, 2, "offsets", "interval")
    rng = np.random.default_rng(n)
    w = (rng.standard_normal((T + 1, n, n)), rng.standard_normal((T + 1, n)), rng.standard_normal(T + 1),
         rng.standard_normal((T + 1, n)), 1.3)
    a = gpu_grads(p, *w)
    p.F = W.Coef(np.repeat(p.F.values, T, axis=0), W.PER_INTERVAL)
    b = gpu_grads(p, *w)
    b["F"] = b["F"].sum(axis=0, keepdims=True)
    for k in a:
        assert grel(a[k], b[k]) <= GTOL, k
