"""Combinations of n = 16 and 64 elements whose states are in mixed units, x = D
x' with D a diagonal of powers of two: an FP64 fold does not feel D in its
products, and neither may the split products (csrc/lqt_split.cuh).  Results are
compared in the units x' with the oracle on the problem in those units.

Bounds: an FP64 fold of these elements leaves at most 1.5e-15 of S and 6e-15 of
v at ratios up to 2^34 on the CPU; 64 times that.  The whole solves are held to
the parity tests' 1e-9.  (From 2^40 on the pivots of I + C J are reported as
SINGULAR.)"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import TOL, relerr as rel, to_np
from tests.test_gpu_split import elements

pytestmark = pytest.mark.gpu


def units(n, ratio, seed, shift=0):
    """n powers of two spread evenly over 2^(-ratio/2) .. 2^(ratio/2), in no order, times 2^shift."""
    e = np.round(np.linspace(-ratio / 2, ratio / 2, n)) + shift
    return 2.0 ** np.random.default_rng(seed).permutation(e)


def in_units(p, D):
    """The problem in the states x = D x'."""
    s = lambda c, f: dataclasses.replace(c, values=f(c.values))
    return dataclasses.replace(
        p, F=s(p.F, lambda v: v * D[:, None] / D[None, :]), L=s(p.L, lambda v: v * D[:, None]),
        X=s(p.X, lambda v: v / np.outer(D, D)), r=s(p.r, lambda v: v * D), Xf=p.Xf / np.outer(D, D), rf=p.rf * D,
        x0=p.x0 * D)


# ratio of units, common factor: 2^-505 brings C to the smallest normal
# numbers and J to the largest
@pytest.mark.parametrize("ratio,shift", [(4, 0), (20, 0), (28, 0), (34, 0), (0, -505), (12, -500)])
@pytest.mark.parametrize("n,T", [(16, 1), (16, 37), (16, 130), (64, 5), (64, 37)])
def test_scan_of_values(n, T, ratio, shift):
    m = __import__("paper_2212_11744_gb300")
    p = W.batched_member(7, T=T, n=16) if n == 16 else W.large_state_n64(T=T)
    el, D = elements(n, T, 100 * T + n), units(n, ratio, T + ratio, shift)
    g = dict(el, A=el["A"] * D[:, None] / D[None, :], C=el["C"] * np.outer(D, D), J=el["J"] / np.outer(D, D),
             b=el["b"] * D, eta=el["eta"] / D)
    out = m.lqt_scan_value(m.DeviceProblem(p), {k: torch.tensor(np.ascontiguousarray(v), device="cuda")
                                                for k, v in g.items()})
    torch.cuda.synchronize()
    assert m.lqt_get_status() == 0
    S, v, _ = oracle.suffix_values(n, el)
    assert rel(to_np(out["S"]) * np.outer(D, D), S) <= 64 * 1.5e-15
    assert rel(to_np(out["v"]) * D, v) <= 64 * 6e-15


@pytest.mark.parametrize("n,T", [(16, 40), (16, 600), (64, 40), (64, 200)])
@pytest.mark.parametrize("method2", [False, True])
def test_solve(n, T, method2):
    m = __import__("paper_2212_11744_gb300")
    p = W.batched_member(5, T=T, n=16) if n == 16 else W.large_state_n64(T=T)
    D = units(n, 34, n + T)
    dp = m.DeviceProblem(in_units(p, D))
    out = m.lqt_solve_method2(dp) if method2 else m.lqt_solve(dp)
    torch.cuda.synchronize()
    ref = oracle.solve(p)
    if method2:  # its states differ from Method 1's by the RK4 error
        ref.update(oracle.trajectory_method2(p, ref["S"], ref["v"]))
    got = {"S": to_np(out["S"]) * np.outer(D, D), "v": to_np(out["v"]) * D, "x": to_np(out["x"]) / D,
           "u": to_np(out["u"])}
    for k, v in got.items():
        assert rel(v, ref[k]) <= TOL, k


@pytest.mark.parametrize("chunk", [0, 2, 8, 32])
def test_batch(chunk):
    from paper_2212_11744_gb300.batch import Batch
    ps = [W.batched_member(40 + i, T=T, n=16) for i, T in enumerate((1, 37, 64, 200, 5))]
    Ds = [units(16, 34 if i % 2 else 0, i) for i in range(len(ps))]
    b = Batch([in_units(p, D) for p, D in zip(ps, Ds)])
    out = b.solve(chunk=chunk)
    torch.cuda.synchronize()
    for i, (p, D) in enumerate(zip(ps, Ds)):
        ref, got = oracle.solve(p), b.problem_slice(out, i)
        assert rel(to_np(got["S"]) * np.outer(D, D), ref["S"]) <= TOL, i
        assert rel(to_np(got["x"]) / D, ref["x"]) <= TOL, i
        assert rel(to_np(got["u"]), ref["u"]) <= TOL, i
