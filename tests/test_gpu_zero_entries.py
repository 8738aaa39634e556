"""The right-hand sides that skip zero entries of a constant F, and those that take
F whole (n = 8, densification): the sums and their order are the same, so the
results are the same bits as with the same F given per sub-interval, where every
entry counts.  F from empty to full, on both sides of the line (7/8 of the entries)."""
import dataclasses

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def lqt():
    import paper_2212_11744_gb300 as m
    return m


def problem(n, m, T, entries, seed):
    """An uneven grid (the general build) and F with so many nonzero entries."""
    rng = np.random.default_rng(seed)
    p = W.batched_member(seed, T=T, n=n)
    F = np.zeros(n * n)
    F[rng.permutation(n * n)[:entries]] = rng.standard_normal(entries) / np.sqrt(n)
    G = rng.standard_normal((m, m))
    d = 0.02 * rng.uniform(0.5, 1.5, T)
    return dataclasses.replace(p, m=m, K=2, F=W.const(F.reshape(n, n)), L=W.const(rng.standard_normal((n, m))),
                               U=W.const(G @ G.T + 0.3 * np.eye(m)), t=np.concatenate([[0.0], np.cumsum(d)]))


def per_interval(p):
    return dataclasses.replace(p, F=W.Coef(np.repeat(p.F.values, p.T, axis=0), W.PER_INTERVAL))


@pytest.mark.parametrize("m", [1, 3, 8])
@pytest.mark.parametrize("entries", [0, 9, 55, 56, 64])
def test_elements_n8(m, entries):
    p = problem(8, m, 24576, entries, 10 * m + entries)  # from 24576 on: one thread per element
    a = lqt().lqt_build_elements(lqt().DeviceProblem(p))
    b = lqt().lqt_build_elements(lqt().DeviceProblem(per_interval(p)))
    torch.cuda.synchronize()
    assert lqt().lqt_get_status() == 0
    for k in ("A", "b", "C", "eta", "J", "zeta"):
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("n,m,entries", [(1, 1, 0), (1, 1, 1), (2, 1, 1), (2, 2, 4), (3, 1, 7), (3, 2, 8), (4, 2, 2),
                                         (4, 4, 13), (4, 1, 14), (8, 4, 9), (8, 1, 55), (8, 8, 64)])
def test_dense_output(n, m, entries):
    p = problem(n if n != 1 and n != 3 else n + 1, m, 259, entries, n + m + entries)
    if n in (1, 3):
        cut = lambda c: W.const(np.ascontiguousarray(c.values[0][:n, :n]))
        F = np.zeros(n * n)
        F[:entries] = np.random.default_rng(n).standard_normal(entries)
        p = dataclasses.replace(p, n=n, nr=n, F=W.const(F.reshape(n, n)), L=W.const(p.L.values[0][:n]), X=cut(p.X),
                                r=W.Coef(p.r.values[:, :n].copy(), p.r.mode), Xf=p.Xf[:n, :n].copy(), rf=p.rf[:n],
                                x0=p.x0[:n])
    dp, dq = lqt().DeviceProblem(p), lqt().DeviceProblem(per_interval(p))
    sol = lqt().lqt_solve(dp)
    a, b = lqt().lqt_densify(dp, sol), lqt().lqt_densify(dq, sol)
    torch.cuda.synchronize()
    assert lqt().lqt_get_status() == 0
    for k in a:
        assert torch.equal(a[k], b[k]), k
